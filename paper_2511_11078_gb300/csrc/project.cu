// project.cu -- forward projection A (Algorithm 2, Eq. 4) and its matched
// adjoint A^T (Sec. 2.3: the same matrix, to FP32 rounding), exact quadrature
// footprint: dispatch, and the forms that need no scratch.
//
// Forward of degrees 1 to 3 with the geometry's scratch: line.cu.  Without it
// (degree 0, captured calls, geometries not prepared): one thread per ray; the 128 threads of a block cover a 16 x 8
// detector tile of one view (a warp is an 8 x 4 sub-tile), so neighbouring
// lanes walk neighbouring lines and gather neighbouring coefficients (L1
// hits).  Each ray is walked with the cell march (one Gauss node set per
// point of the ray, an (n+1)^3 register window); the per-cell partial sums
// are added along the ray with Kahan compensation.
//
// Adjoint, view geometries, two forms that visit the same pairs with the
// same footprints:
//  * scatter (default, scatter.cu): the forward's thread mapping, vector
//    reductions into layouts of c; flat parallel views reduce into c here;
//  * gather: one block per 16^3 coefficient brick; for every batch of 8
//    views the block projects the brick's support box onto the detectors,
//    walks the rays of those pixel windows through the brick's cells with
//    the piece march, accumulates y_r * P in shared memory and folds the
//    batch into FP64 totals; no global atomics, each coefficient written
//    once.
// Adjoint, explicit rays: no view structure to gather over: scatter.
#include <stdio.h>
#include <string.h>

#include "spl_host.h"
#include "spl_mlp.cuh"

namespace spl {

// ---------------------------------------------------------------- sinks
// Sinks take a basis either by index (flush, the flat cell march) or by its
// offset in the sink's layout, off + l_d S0 + l_a S1 + l_b S2 in unsigned
// (wrapping) arithmetic, with a flag that it lies in the region (put, the
// piece march).
struct FwdSink {
    static constexpr bool plane = false;
    const float *__restrict__ c;
    int S0, S1, S2;
    unsigned off;
    SinkBox bx;
    float inv_wd;
    bool kahan;
    // the cell's partial sum c_l * F_l, spread over four independent
    // accumulators (a face's 16 gathers and FMAs then form four chains of
    // four instead of one chain of sixteen)
    float acc[4], sum, comp;
    __device__ __forceinline__ void piece() {}
    __device__ __forceinline__ bool relevant(int d0, int d1, int a0, int a1, int b0, int b1) const
    {
        return bx.meets(d0, d1, a0, a1, b0, b1);
    }
    __device__ __forceinline__ void flush(int ld, int la, int lb, float v)
    {
        if (bx.holds(ld, la, lb)) acc[0] = fmaf(__ldg(c + (ld * S0 + la * S1 + lb * S2)), v, acc[0]);
    }
    __device__ __forceinline__ void put(unsigned o, bool in, float v, int slot)
    {
        if (in) acc[slot & 3] = fmaf(__ldg(c + o), v, acc[slot & 3]);
    }
    __device__ __forceinline__ void cell_end()
    {
        const float v = ((acc[0] + acc[1]) + (acc[2] + acc[3])) * inv_wd;
        acc[0] = acc[1] = acc[2] = acc[3] = 0.0f;
        if (kahan) kahan_add(sum, comp, v);
        else sum += v;
    }
};

struct CountSink {
    static constexpr bool plane = false;
    int S0, S1, S2;
    unsigned off;
    SinkBox bx;
    unsigned int n;       // bases with a nonzero footprint
    unsigned int pieces;  // integrated pieces (GL nodes each)
    __device__ __forceinline__ void piece() { ++pieces; }
    __device__ __forceinline__ bool relevant(int d0, int d1, int a0, int a1, int b0, int b1) const
    {
        return bx.meets(d0, d1, a0, a1, b0, b1);
    }
    __device__ __forceinline__ void flush(int ld, int la, int lb, float v)
    {
        n += (bx.holds(ld, la, lb) && v > 0.0f) ? 1u : 0u;
    }
    __device__ __forceinline__ void put(unsigned, bool in, float v, int) { n += (in && v > 0.0f) ? 1u : 0u; }
    __device__ __forceinline__ void cell_end() {}
};

// adjoint, flat parallel views: y_r / |w_d| * F_l added to c_l with a float
// atomic
struct AtomicSink {
    static constexpr bool plane = false;
    float *__restrict__ c;
    int S0, S1, S2;
    SinkBox bx;
    float yv;
    __device__ __forceinline__ void piece() {}
    __device__ __forceinline__ bool relevant(int d0, int d1, int a0, int a1, int b0, int b1) const
    {
        return bx.meets(d0, d1, a0, a1, b0, b1);
    }
    __device__ __forceinline__ void flush(int ld, int la, int lb, float v)
    {
        if (bx.holds(ld, la, lb)) atomicAdd(c + (ld * S0 + la * S1 + lb * S2), yv * v);
    }
    __device__ __forceinline__ void cell_end() {}
};

// brick of the gather adjoint: the region is the brick, the target the
// shared-memory brick array (mirrored strides S0..S2, offset off)
struct BrickSink {
    static constexpr bool plane = false;
    float *part;
    int S0, S1, S2;
    unsigned off;
    SinkBox bx;
    float yv;
    __device__ __forceinline__ void piece() {}
    __device__ __forceinline__ bool relevant(int d0, int d1, int a0, int a1, int b0, int b1) const
    {
        return bx.meets(d0, d1, a0, a1, b0, b1);
    }
    __device__ __forceinline__ void flush(int ld, int la, int lb, float v)
    {
        if (bx.holds(ld, la, lb)) atomicAdd(part + (unsigned)(ld * S0 + la * S1 + lb * S2 + (int)off), yv * v);
    }
    __device__ __forceinline__ void put(unsigned o, bool in, float v, int)
    {
        if (in) atomicAdd(part + o, yv * v);
    }
    __device__ __forceinline__ void cell_end() {}
};

// ---------------------------------------------------------------- forward

// View classes of a view-kernel launch.  VM_FLAT / VM_GENERAL: parallel
// views of one class, taken from the geometry's view order; the form is
// fixed at compile time, so each kernel carries the registers of one form
// only (a parallel view's rays share their direction, hence their form).
// VM_CONE: cone views, every ray with the piece march (a cone ray with a
// zero direction component, rare, is integrated by the general form too:
// its constant factor is then evaluated at every node, which is exact but
// slower; the kernel keeps the registers and code of one form).  VM_RAYS:
// explicit rays, the form chosen per ray.
enum { VM_CONE = 0, VM_FLAT = 1, VM_GENERAL = 2, VM_RAYS = 3 };

template <int N, int VM, class Sink>
__device__ __forceinline__ bool march_vm(const RaySetup &rs, int cf, int cl, const QuadRule &qr, Sink &sk)
{
    if constexpr (VM == VM_FLAT) return cell_march<N, Sink, true>(rs, cf, cl, qr, sk);
    else if constexpr (VM == VM_GENERAL || VM == VM_CONE) return piece_march<N, Sink>(rs, cf, cl, qr, sk);
    else return march<N>(rs, cf, cl, qr, sk);
}

// The march form of a ray of geometry kind `kind` (used where one kernel
// serves every view kind: the pair count and the brick adjoint), the same
// as the projection kernels': cone rays always take the piece march.
template <int N, class Sink>
__device__ __forceinline__ bool march_kind(int kind, const RaySetup &rs, int cf, int cl, const QuadRule &qr, Sink &sk)
{
    if (kind == SPL_CONE) return piece_march<N, Sink>(rs, cf, cl, qr, sk);
    return march<N>(rs, cf, cl, qr, sk);
}

// blocks per SM the register budget is sized for (measured): the flat form
// needs an (n+1)^2 window, the general one (n+1)^3 accumulators plus the
// flush state (3 blocks x 168 registers; 4 x 128 spills and is slower); the
// direct march keeps (n+1)^3 coefficients but no flush state (4 x 128)
template <int VM, bool DIRECT = false> struct ViewBlocks {
    static constexpr int value = VM == VM_FLAT ? 6 : (DIRECT ? 4 : 3);
};

// DIRECT: rays with three nonzero direction components take the direct
// march (the line integral of f itself); flat rays keep the footprint form
template <int N, int VM, bool DIRECT = false>
__device__ __forceinline__ float march_forward(const RaySetup &rs, const float *__restrict__ c, const QuadRule &qr,
                                               bool kahan, int *err)
{
    if constexpr (DIRECT && VM != VM_FLAT) {
        if (VM == VM_GENERAL || VM == VM_CONE || rs.rb != 0.0f) {
            float out;
            if (!direct_march<N>(rs, c, rs.S[0], rs.S[1], rs.S[2], make_box(rs.lo, rs.hi), qr, kahan, out))
                atomicOr(err, 1);
            return out;
        }
    }
    FwdSink sk;
    sk.c = c;
    sk.S0 = rs.S[0];
    sk.S1 = rs.S[1];
    sk.S2 = rs.S[2];
    sk.off = 0u;
    sk.bx = make_box(rs.lo, rs.hi);
    sk.inv_wd = rs.inv_wd;
    sk.kahan = kahan;
    sk.acc[0] = sk.acc[1] = sk.acc[2] = sk.acc[3] = sk.sum = sk.comp = 0.0f;
    if (!march_vm<N, VM>(rs, rs.c0, rs.c1, qr, sk)) atomicOr(err, 1);
    return sk.sum;
}

// cone views (every ray with the piece march)
template <int N, bool DIRECT>
__global__ void __launch_bounds__(128, (ViewBlocks<VM_CONE, DIRECT>::value))
    k_forward_views(DevGeom g, const float *__restrict__ c, float *__restrict__ y, QuadRule qr, int kahan)
{
    int iu, iv;
    tile_pixel(iu, iv);
    const int k = blockIdx.z;
    if (iu >= g.nu || iv >= g.nv) return;
    RaySetup rs;
    float v = 0.0f;
    if (view_setup<N>(g, grid_of(g), k, iu, iv, rs))
        v = march_forward<N, VM_CONE, DIRECT>(rs, c, qr, kahan != 0, g.err);
    y[((long long)k * g.nv + iv) * g.nu + iu] = v;
}

// parallel views of one class (VM_FLAT or VM_GENERAL): view blockIdx.z of
// the chunk
template <int N, int VM, bool DIRECT>
__global__ void __launch_bounds__(128, (ViewBlocks<VM, DIRECT>::value))
    k_forward_pviews(DevGeom g, const float *__restrict__ c, float *__restrict__ y, QuadRule qr, int kahan,
                     const __grid_constant__ ViewChunk vc)
{
    int iu, iv;
    tile_pixel(iu, iv);
    const ViewConst &V = vc.v[blockIdx.z];
    const int k = V.view;
    if (iu >= g.nu || iv >= g.nv) return;
    RaySetup rs;
    float v = 0.0f;
    if (view_setup<N>(g, grid_of(g), k, iu, iv, rs)) {
        use_view_const(V, rs);
        v = march_forward<N, VM, DIRECT>(rs, c, qr, kahan != 0, g.err);
    }
    y[((long long)k * g.nv + iv) * g.nu + iu] = v;
}

template <int N, bool DIRECT>
__global__ void __launch_bounds__(128) k_forward_rays(DevGeom g, const float *__restrict__ c, float *__restrict__ y,
                                                      QuadRule qr, int kahan)
{
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= g.n_rays) return;
    double s[3], w[3];
    explicit_ray(g, r, s, w);
    RaySetup rs;
    float v = 0.0f;
    if (ray_setup<N>(grid_of(g), s, w, rs)) v = march_forward<N, VM_RAYS, DIRECT>(rs, c, qr, kahan != 0, g.err);
    y[r] = v;
}

// ---------------------------------------------------------------- pair count
template <int N>
__device__ __forceinline__ void march_count(int kind, const RaySetup &rs, const QuadRule &qr, int *err,
                                            unsigned int &pairs, unsigned int &pieces, unsigned int &flat_pieces)
{
    CountSink sk;
    sk.S0 = sk.S1 = sk.S2 = 0;
    sk.off = 0u;
    sk.bx = make_box(rs.lo, rs.hi);
    sk.n = 0u;
    sk.pieces = 0u;
    if (!march_kind<N>(kind, rs, rs.c0, rs.c1, qr, sk)) atomicOr(err, 1);
    const bool flat = rs.rb == 0.0f && kind != SPL_CONE;
    pairs = sk.n;  // (nonzero FP32 footprints; the contributions come from the exact count)
    pieces = flat ? 0u : sk.pieces;
    flat_pieces = flat ? sk.pieces : 0u;
}

__device__ __forceinline__ void add_count(unsigned long long *count, unsigned int v)
{
    unsigned long long x = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(count, x);
}

template <int N>
__global__ void __launch_bounds__(128) k_count_views(DevGeom g, unsigned long long *count, QuadRule qr)
{
    int iu, iv;
    tile_pixel(iu, iv);
    const int k = blockIdx.z;
    unsigned int v = 0, pc = 0, pf = 0;
    RaySetup rs;
    if (iu < g.nu && iv < g.nv && view_setup<N>(g, grid_of(g), k, iu, iv, rs))
        march_count<N>(g.kind, rs, qr, g.err, v, pc, pf);
    add_count(count + 1, pc);
    add_count(count + 2, pf);
}

template <int N>
__global__ void __launch_bounds__(128) k_count_rays(DevGeom g, unsigned long long *count, QuadRule qr)
{
    const long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned int v = 0, pc = 0, pf = 0;
    if (r < g.n_rays) {
        double s[3], w[3];
        explicit_ray(g, r, s, w);
        RaySetup rs;
        if (ray_setup<N>(grid_of(g), s, w, rs)) march_count<N>(SPL_RAYS, rs, qr, g.err, v, pc, pf);
    }
    add_count(count + 1, pc);
    add_count(count + 2, pf);
}

// ---------------------------------------------------------------- adjoint: flat parallel views
// The flat views outside the plane group: the forward's thread mapping, the
// flat cell march, scalar atomics into c.  Every other ray scatters through
// scatter.cu.
template <int N>
__global__ void __launch_bounds__(128, ViewBlocks<VM_FLAT>::value)
    k_adjoint_flat_scatter(DevGeom g, const float *__restrict__ y, float *__restrict__ c, QuadRule qr,
                           const __grid_constant__ ViewChunk vc)
{
    int iu, iv;
    tile_pixel(iu, iv);
    const ViewConst &V = vc.v[blockIdx.z];
    const int k = V.view;
    if (iu >= g.nu || iv >= g.nv) return;
    const float yr = __ldg(y + ((long long)k * g.nv + iv) * g.nu + iu);
    if (yr == 0.0f) return;
    RaySetup rs;
    if (!view_setup<N>(g, grid_of(g), k, iu, iv, rs)) return;
    use_view_const(V, rs);
    AtomicSink sk;
    sk.c = c;
    sk.S0 = rs.S[0];
    sk.S1 = rs.S[1];
    sk.S2 = rs.S[2];
    sk.bx = make_box(rs.lo, rs.hi);
    sk.yv = yr * rs.inv_wd;
    if (!cell_march<N, AtomicSink, true>(rs, rs.c0, rs.c1, qr, sk)) atomicOr(g.err, 1);
}

// ---------------------------------------------------------------- adjoint: brick gather (view geometries)
constexpr int kBrick = 16;                        // brick edge (coefficients)
constexpr int kBrickVol = kBrick * kBrick * kBrick;
constexpr int kAdjThreads = 256;
constexpr int kViewBatch = 8;                     // views per shared-memory fold

// detector pixel window of the box [lo, hi] (world) for view k: projection
// of its 8 corners (parallel: along the direction; cone: from the source)
__device__ __forceinline__ bool pixel_window(const DevGeom &g, int k, const double (&lo)[3], const double (&hi)[3],
                                             int &u0, int &u1, int &v0, int &v1)
{
    const ViewPose &P = g.views[k];
    double amin = 1e300, amax = -1e300, bmin = 1e300, bmax = -1e300;
    const double cu = 0.5 * (g.nu - 1), cv = 0.5 * (g.nv - 1);
#pragma unroll
    for (int corner = 0; corner < 8; ++corner) {
        double x[3] = {(corner & 1) ? hi[0] : lo[0], (corner & 2) ? hi[1] : lo[1], (corner & 4) ? hi[2] : lo[2]};
        double pt[3];
        if (g.kind == 1) {
            // move x along the direction onto the detector plane
            double rel[3] = {x[0] - P.dc[0], x[1] - P.dc[1], x[2] - P.dc[2]};
            const double t = (rel[0] * P.nrm[0] + rel[1] * P.nrm[1] + rel[2] * P.nrm[2]) /
                             (P.src[0] * P.nrm[0] + P.src[1] * P.nrm[1] + P.src[2] * P.nrm[2]);
#pragma unroll
            for (int e = 0; e < 3; ++e) pt[e] = rel[e] - t * P.src[e];
        } else {
            double dx[3] = {x[0] - P.src[0], x[1] - P.src[1], x[2] - P.src[2]};
            double sd[3] = {P.dc[0] - P.src[0], P.dc[1] - P.src[1], P.dc[2] - P.src[2]};
            const double num = sd[0] * P.nrm[0] + sd[1] * P.nrm[1] + sd[2] * P.nrm[2];
            const double den = dx[0] * P.nrm[0] + dx[1] * P.nrm[1] + dx[2] * P.nrm[2];
            if (!(den * num > 0.0)) return true;  // corner behind the source: keep the whole detector
            const double lam = num / den;
#pragma unroll
            for (int e = 0; e < 3; ++e) pt[e] = P.src[e] + lam * dx[e] - P.dc[e];
        }
        const double a = pt[0] * P.ud[0] + pt[1] * P.ud[1] + pt[2] * P.ud[2];
        const double b = pt[0] * P.vd[0] + pt[1] * P.vd[1] + pt[2] * P.vd[2];
        amin = fmin(amin, a);
        amax = fmax(amax, a);
        bmin = fmin(bmin, b);
        bmax = fmax(bmax, b);
    }
    // clamp to the detector before converting (far corners stay in range)
    const double eps = 1e-3;
    u0 = (int)fmin(fmax(0.0, ceil(amin + cu - eps)), (double)g.nu);
    u1 = (int)fmax(fmin((double)(g.nu - 1), floor(amax + cu + eps)), -1.0);
    v0 = (int)fmin(fmax(0.0, ceil(bmin + cv - eps)), (double)g.nv);
    v1 = (int)fmax(fmin((double)(g.nv - 1), floor(bmax + cv + eps)), -1.0);
    return false;
}

// Clip the cell range [cf, cl] of a ray to the cells whose window can hold a
// basis of the brick: over cell c the window's a-range is
// [floor(v_a(c)) - N, floor(v_a(c+1))], v_a(c) = V + (c - c0) r_a (same for
// b).  Conservative by two cells; starting before the first such cell is
// what keeps the brick's values equal to the full march's.
template <int N>
__device__ __forceinline__ void clip_cells_to_brick(const RaySetup &rs, const int (&blo)[3], const int (&bhi)[3],
                                                    int &cf, int &cl)
{
    const float base[2] = {rs.Vah + rs.Val, rs.Vbh + rs.Vbl};
    const float r[2] = {rs.ra, rs.rb}, ir[2] = {rs.inv_ra, rs.inv_rb};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (r[q] > 0.0f) {
            const float cfl = rs.c0 + (blo[q + 1] - base[q]) * ir[q];
            const float chl = rs.c0 + (bhi[q + 1] + N + 1 - base[q]) * ir[q];
            cf = max(cf, (int)fmaxf(floorf(cfl) - 2.0f, -1e9f));
            cl = min(cl, (int)fminf(ceilf(chl) + 1.0f, 1e9f));
        } else if (!(base[q] + 1.0f > blo[q + 1] && base[q] - (N + 1) < bhi[q + 1])) {
            cl = cf - 1;
        }
    }
}

// vlist: the views to walk (NULL: all views 0 .. nview-1); add: c += the
// brick totals instead of c = them
template <int N>
__global__ void __launch_bounds__(kAdjThreads) k_adjoint_bricks(DevGeom g, const float *__restrict__ y,
                                                                float *__restrict__ c, QuadRule qr, int bx, int by,
                                                                const int *vlist, int nview, int add)
{
    extern __shared__ __align__(16) unsigned char smem[];
    double *tot = (double *)smem;                                // kBrickVol FP64 totals
    float *part = (float *)(smem + kBrickVol * sizeof(double));  // kBrickVol partials of a view batch
    __shared__ int win[kViewBatch][3];                           // u0, wu, v0 of each view of the batch
    __shared__ int woff[kViewBatch + 1];                         // prefix sums of the window sizes
    __shared__ int next_item;
    constexpr double W = 0.5 * (N + 1);
    const int bid = blockIdx.x;
    const int b0[3] = {(bid % bx) * kBrick, ((bid / bx) % by) * kBrick, (bid / (bx * by)) * kBrick};
    int bn[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) bn[e] = min(kBrick, g.n[e] - b0[e]);
    for (int i = threadIdx.x; i < kBrickVol; i += kAdjThreads) {
        tot[i] = 0.0;
        part[i] = 0.0f;
    }
    // support box of the brick's bases (world)
    double lo[3], hi[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        lo[e] = g.org[e] + b0[e] - W;
        hi[e] = g.org[e] + b0[e] + bn[e] - 1 + W;
    }
    const GridBox gb = grid_of(g);
    const int lstride[3] = {1, kBrick, kBrick * kBrick};
    bool ok = true;
    __shared__ int vk[kViewBatch];
    for (int k0 = 0; k0 < nview; k0 += kViewBatch) {
        const int nb = min(kViewBatch, nview - k0);
        if (threadIdx.x < nb) {
            const int kv = vlist ? vlist[k0 + threadIdx.x] : k0 + threadIdx.x;
            vk[threadIdx.x] = kv;
            int u0, u1, v0, v1;
            if (pixel_window(g, kv, lo, hi, u0, u1, v0, v1)) {
                u0 = 0;
                u1 = g.nu - 1;
                v0 = 0;
                v1 = g.nv - 1;
            }
            const int wu = u1 - u0 + 1, wv = v1 - v0 + 1;
            win[threadIdx.x][0] = u0;
            win[threadIdx.x][1] = wu > 0 ? wu : 0;
            win[threadIdx.x][2] = v0;
            woff[threadIdx.x + 1] = (wu > 0 && wv > 0) ? wu * wv : 0;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            woff[0] = 0;
            for (int t = 1; t <= nb; ++t) woff[t] += woff[t - 1];
            next_item = 0;
        }
        __syncthreads();
        const int total = woff[nb];
        // rays are taken one at a time from a shared counter: their costs
        // differ a lot (a ray may cross one slab of the brick or sixteen)
        for (int item = atomicAdd(&next_item, 1); item < total; item = atomicAdd(&next_item, 1)) {
            int t = 0;
            while (item >= woff[t + 1]) ++t;
            const int p = item - woff[t];
            const int iu = win[t][0] + p % win[t][1], iv = win[t][2] + p / win[t][1];
            const int k = vk[t];
            const float yr = __ldg(y + ((long long)k * g.nv + iv) * g.nu + iu);
            if (yr == 0.0f) continue;
            RaySetup rs;
            if (!view_setup<N>(g, gb, k, iu, iv, rs)) continue;
            // brick bounds in the ray's mirrored (d, a, b) coordinates
            int blo[3], bhi[3], L[3], Loff = 0;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int e = rs.ax[q];
                const int r0 = b0[e], r1 = b0[e] + bn[e] - 1;
                blo[q] = rs.sg[q] > 0 ? r0 : -r1;
                bhi[q] = rs.sg[q] > 0 ? r1 : -r0;
                L[q] = rs.sg[q] * lstride[e];
                Loff -= b0[e] * lstride[e];
            }
            // a brick basis l_d is live in cells l_d .. l_d + N
            int cf = max(rs.c0, blo[0]), cl = min(rs.c1, bhi[0] + N);
            clip_cells_to_brick<N>(rs, blo, bhi, cf, cl);
            if (cf > cl) continue;
            BrickSink sk;
            sk.part = part;
            sk.S0 = L[0];
            sk.S1 = L[1];
            sk.S2 = L[2];
            sk.off = (unsigned)Loff;
            sk.bx = make_box(blo, bhi);
            sk.yv = yr * rs.inv_wd;
            ok &= march_kind<N>(g.kind, rs, cf, cl, qr, sk);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kBrickVol; i += kAdjThreads) {
            tot[i] += (double)part[i];
            part[i] = 0.0f;
        }
        __syncthreads();
    }
    if (!ok) atomicOr(g.err, 1);
    for (int i = threadIdx.x; i < kBrickVol; i += kAdjThreads) {
        const int lx = i % kBrick, ly = (i / kBrick) % kBrick, lz = i / (kBrick * kBrick);
        if (lx < bn[0] && ly < bn[1] && lz < bn[2]) {
            float &dst = c[((long long)(b0[2] + lz) * g.n[1] + (b0[1] + ly)) * g.n[0] + (b0[0] + lx)];
            dst = add ? (float)((double)dst + tot[i]) : (float)tot[i];
        }
    }
}

constexpr size_t kAdjSmem = kBrickVol * (sizeof(double) + sizeof(float));

// Batched scatter: acc += c (FP64 total of the batches), and c = acc at the
// end.  Grid-strided, coalesced.
__global__ void k_acc_add(long long n, double *__restrict__ acc, const float *__restrict__ c)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) acc[i] += (double)c[i];
}

__global__ void k_acc_store(long long n, const double *__restrict__ acc, float *__restrict__ c)
{
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) c[i] = (float)acc[i];
}

}  // namespace spl

using namespace spl;

static spl_status launch_status(const char *what)
{
    return cuda_check(cudaGetLastError(), what);
}

// Launch `launch(chunk, n)` for the parallel views view_order[v0 .. v0+count)
// in chunks of at most `per` (<= kViewChunk) views, each with its views'
// constants.
template <class F>
static void for_view_chunks(const spl_geometry *g, int v0, int count, F launch, int per = kViewChunk)
{
    static thread_local ViewChunk ch;
    for (int s = 0; s < count; s += per) {
        const int n = count - s < per ? count - s : per;
        memcpy(ch.v, g->vconst + v0 + s, (size_t)n * sizeof(ViewConst));
        launch(ch, n);
    }
}

static unsigned stream_grid(long long n)
{
    const long long b = (n + 255) / 256, cap = 8LL * sm_count();
    return (unsigned)(b < cap ? (b > 0 ? b : 1) : cap);
}

// Parallel geometries: the separable group through the plane matrices
// (when used), the other flat views with the flat kernel, the rest with the
// general one.  Returns the first view_order index the flat kernel takes.
// The plane matrices are built by spl_prepare only: unbuilt is an error
// (SPL_ERR_STATE), unavailable (their allocation failed) walks the views.
static int plane_views(const spl_geometry *g, const spl_basis_desc *b, spl_status *err)
{
    *err = SPL_OK;
    if (b->separable == SPL_SEP_OFF || b->mode == SPL_FP_MLP || b->mode == SPL_FP_TABLE || !g->plane) return 0;
    const int state = plane_state(g, b->degree);
    if (state == 0) {
        *err = fail(SPL_ERR_STATE, "plane matrices of degree %d not built: call spl_prepare first", b->degree);
        return 0;
    }
    return state == 1 ? g->dev.n_sep : 0;
}

template <int N, bool DIRECT>
static spl_status forward_quad_t(const spl_geometry *g, const spl_basis_desc *b, const float *c, float *y,
                                 bool captured, cudaStream_t st)
{
    const DevGeom &dg = g->dev;
    const QuadRule qr = quad_rule(N);
    const int kahan = b->kahan;
    const bool line = line_usable(g, N, captured);
    if (line && dg.kind != SPL_PARALLEL) return line_forward(g, N, kahan, c, y, st);
    if (dg.kind == SPL_RAYS) {
        const long long blocks = (dg.n_rays + 127) / 128;
        k_forward_rays<N, DIRECT><<<(unsigned)blocks, 128, 0, st>>>(dg, c, y, qr, kahan);
    } else if (dg.kind == SPL_PARALLEL) {
        spl_status s;
        const int v0 = plane_views(g, b, &s);
        if (s != SPL_OK) return s;
        // the plane path (memory-latency bound) runs beside the march of the
        // other views (arithmetic bound) when both have work: the two write
        // disjoint rows of y
        const bool overlap = v0 > 0 && v0 < dg.n_views && g->plane->side;
        if (v0 > 0) {
            cudaStream_t ps = st;
            if (overlap) {
                s = cuda_check(cudaEventRecord(g->plane->fork, st), "fork record");
                if (s == SPL_OK) s = cuda_check(cudaStreamWaitEvent(g->plane->side, g->plane->fork, 0), "fork wait");
                if (s != SPL_OK) return s;
                ps = g->plane->side;
            }
            s = plane_forward(g, N, kahan, c, y, ps);
            if (overlap) {
                const spl_status sj = cuda_check(cudaEventRecord(g->plane->join, ps), "join record");
                if (s != SPL_OK || sj != SPL_OK) {
                    // join the side stream before returning the error, so the
                    // caller's stream (or its graph capture) never leaves it
                    // unjoined
                    if (sj == SPL_OK) cudaStreamWaitEvent(st, g->plane->join, 0);
                    return s != SPL_OK ? s : sj;
                }
            }
            if (s != SPL_OK) return s;
        }
        const unsigned gx = (dg.nu + 15) / 16, gy = (dg.nv + 7) / 8;
        for_view_chunks(g, v0, dg.n_flat - v0, [&](const ViewChunk &ch, int n) {
            k_forward_pviews<N, VM_FLAT, false><<<dim3(gx, gy, n), 128, 0, st>>>(dg, c, y, qr, kahan, ch);
        });
        if (line) s = line_forward(g, N, kahan, c, y, st);
        else for_view_chunks(g, dg.n_flat, dg.n_views - dg.n_flat, [&](const ViewChunk &ch, int n) {
            k_forward_pviews<N, VM_GENERAL, DIRECT><<<dim3(gx, gy, n), 128, 0, st>>>(dg, c, y, qr, kahan, ch);
        });
        if (overlap) {
            const spl_status sj = cuda_check(cudaStreamWaitEvent(st, g->plane->join, 0), "join wait");
            if (s == SPL_OK) s = sj;
        }
        if (s != SPL_OK) return s;
    } else {
        dim3 grid((dg.nu + 15) / 16, (dg.nv + 7) / 8, dg.n_views);
        k_forward_views<N, DIRECT><<<grid, 128, 0, st>>>(dg, c, y, qr, kahan);
    }
    return launch_status("forward launch");
}

template <int N>
static spl_status forward_quad(const spl_geometry *g, const spl_basis_desc *b, const float *c, float *y, cudaStream_t st)
{
    if (g->dev.n_rays == 0) return SPL_OK;
    auto run = [&](bool captured) {
        return b->mode == SPL_FP_DIRECT ? forward_quad_t<N, true>(g, b, c, y, captured, st)
                                        : forward_quad_t<N, false>(g, b, c, y, captured, st);
    };
    ForwardTurn *t = g->turn;
    if (!t) return run(false);
    if (stream_captures(st)) return run(true);
    std::lock_guard<std::mutex> lock(t->mu);
    spl_status s = t->used ? cuda_check(cudaStreamWaitEvent(st, t->last, 0), "forward turn wait") : SPL_OK;
    if (s != SPL_OK) return s;
    s = run(false);
    // recorded also after a failure: what did start still uses the scratch
    const spl_status e = cuda_check(cudaEventRecord(t->last, st), "forward turn record");
    t->used = true;
    return s != SPL_OK ? s : e;
}

// The scatter form over the views from v0 of the view order (or all rays):
// the flat class into c, the rest into the layout copies (scatter.cu).
// has_c: c already holds a part of the result.
//
// Both add y_r * F_l with FP32 atomics.  A coefficient of a large geometry
// receives tens of thousands of them (512^3 helical: ~4e4), and an FP32
// running sum of that many terms loses ~1e-5 of its value; so a geometry with
// more than one batch of views (rays) adds each batch to an FP64 total (its
// scratch, acc64, is allocated with the geometry), which is rounded to c with
// the last batch.  Each batch's FP32 sum has ~1/B of the terms and of the
// magnitude, so its rounding error is ~1/B of the whole.
template <int N>
static spl_status adjoint_scatter(const spl_geometry *g, const float *y, float *c, int v0, bool has_c, const QuadRule &qr,
                                  cudaStream_t st)
{
    const DevGeom &dg = g->dev;
    const long long nc = (long long)dg.n[0] * dg.n[1] * dg.n[2];
    const bool batched = g->acc64 != nullptr, par = dg.kind == SPL_PARALLEL;
    const long long i0 = par ? dg.n_flat : 0, i1 = dg.kind == SPL_RAYS ? dg.n_rays : dg.n_views;
    const bool flat = par && v0 < dg.n_flat, rest = dg.n_rays > 0 && i0 < i1;
    spl_status s = SPL_OK;
    bool has_total = false;  // the FP64 total holds a part of the result
    auto clear_c = [&]() {
        if (s == SPL_OK) s = cuda_check(cudaMemsetAsync(c, 0, nc * sizeof(float), st), "adjoint clear");
    };
    auto add_c = [&]() {  // total += c
        if (s == SPL_OK && !has_total)
            s = cuda_check(cudaMemsetAsync(g->acc64, 0, nc * sizeof(double), st), "adjoint accumulator clear");
        if (s != SPL_OK) return;
        has_total = true;
        k_acc_add<<<stream_grid(nc), 256, 0, st>>>(nc, g->acc64, c);
    };
    if (batched && has_c && (flat || rest)) add_c();
    if (flat) {
        const unsigned gx = (dg.nu + 15) / 16, gy = (dg.nv + 7) / 8;
        if (!batched && !has_c) clear_c();
        for_view_chunks(g, v0, dg.n_flat - v0, [&](const ViewChunk &ch, int n) {
            if (batched) clear_c();
            if (s != SPL_OK) return;
            k_adjoint_flat_scatter<N><<<dim3(gx, gy, n), 128, 0, st>>>(dg, y, c, qr, ch);
            if (batched) add_c();
        }, batched ? kAdjBatchViews : kViewChunk);
        has_c = true;
    }
    long long per = !batched ? i1 : (dg.kind == SPL_RAYS ? kAdjBatchRays : kAdjBatchViews);
    if (batched && dg.kind == SPL_RAYS && scatter_batch(g, N) < per) per = scatter_batch(g, N);
    for (long long i = i0; rest && i < i1 && s == SPL_OK; i += per) {
        const bool last = i + per >= i1;
        s = scatter_rays(g, N, y, i, last ? i1 : i + per, st);
        if (s != SPL_OK) break;
        s = scatter_fold(g, N, has_total ? 2 : (has_c && !batched ? 1 : 0), batched && !last, c, st);
        has_total = has_total || (batched && !last);
    }
    if (s != SPL_OK) return s;
    if (!rest && has_total) k_acc_store<<<stream_grid(nc), 256, 0, st>>>(nc, g->acc64, c);
    else if (!rest && !has_c) clear_c();
    return s == SPL_OK ? launch_status("adjoint launch") : s;
}

template <int N>
static spl_status adjoint_quad(const spl_geometry *g, const spl_basis_desc *b, const float *y, float *c, cudaStream_t st)
{
    const DevGeom &dg = g->dev;
    const QuadRule qr = quad_rule(N);
    const int form = b->adjoint;
    const long long nc = (long long)dg.n[0] * dg.n[1] * dg.n[2];
    spl_status s = SPL_OK;
    int v0 = 0;
    if (dg.kind == SPL_PARALLEL) {
        v0 = plane_views(g, b, &s);
        if (s != SPL_OK) return s;
    }
    const bool scatter = dg.kind == SPL_RAYS || form != SPL_ADJ_GATHER;
    // With the scatter form the plane path's gather (T, memory-latency
    // bound) runs on the geometry's side stream beside the scatter of the
    // other views (arithmetic bound); after the join, T's contribution is
    // added to c.  Otherwise the plane path writes every coefficient first
    // and the other views add.
    const bool overlap = dg.n_rays > 0 && v0 > 0 && v0 < dg.n_views && scatter && g->plane->side;
    if (overlap) {
        s = cuda_check(cudaEventRecord(g->plane->fork, st), "fork record");
        if (s == SPL_OK) s = cuda_check(cudaStreamWaitEvent(g->plane->side, g->plane->fork, 0), "fork wait");
        if (s != SPL_OK) return s;
        s = plane_adjoint_t(g, N, y, g->plane->side);
        const spl_status sj = cuda_check(cudaEventRecord(g->plane->join, g->plane->side), "join record");
        if (s == SPL_OK && sj == SPL_OK) s = adjoint_scatter<N>(g, y, c, v0, false, qr, st);
        // join the side stream also on an error
        const spl_status sw =
            sj == SPL_OK ? cuda_check(cudaStreamWaitEvent(st, g->plane->join, 0), "join wait") : sj;
        if (s == SPL_OK) s = sw;
        return s == SPL_OK ? plane_adjoint_add(g, N, c, st) : s;
    }
    if (v0 > 0) {
        s = plane_adjoint(g, N, y, c, st);
        if (s != SPL_OK) return s;
    }
    if (scatter) return adjoint_scatter<N>(g, y, c, v0, v0 > 0, qr, st);
    if (dg.n_rays == 0) return cuda_check(cudaMemsetAsync(c, 0, nc * sizeof(float), st), "adjoint clear");
    s = smem_attr_once((const void *)k_adjoint_bricks<N>, (int)kAdjSmem, "adjoint smem attribute");
    if (s != SPL_OK) return s;
    const int bx = (dg.n[0] + kBrick - 1) / kBrick, by = (dg.n[1] + kBrick - 1) / kBrick,
              bz = (dg.n[2] + kBrick - 1) / kBrick;
    // bricks over the views the plane path did not take (all of them
    // without it); with the plane path they add to its result
    const int *vlist = v0 > 0 ? dg.view_order + v0 : nullptr;
    const int nview = dg.n_views - v0;
    k_adjoint_bricks<N><<<bx * by * bz, kAdjThreads, kAdjSmem, st>>>(dg, y, c, qr, bx, by, vlist, nview, v0 > 0 ? 1 : 0);
    return launch_status("adjoint launch");
}

template <int N>
static spl_status count_pairs(const spl_geometry *g, unsigned long long *count, cudaStream_t st)
{
    const DevGeom &dg = g->dev;
    const QuadRule qr = quad_rule(N);
    if (dg.n_rays == 0) return SPL_OK;
    spl_status s = count_exact(g, N, count, nullptr, st);
    if (s != SPL_OK) return s;
    if (dg.kind == SPL_RAYS) {
        const long long blocks = (dg.n_rays + 127) / 128;
        k_count_rays<N><<<(unsigned)blocks, 128, 0, st>>>(dg, count, qr);
    } else {
        dim3 grid((dg.nu + 15) / 16, (dg.nv + 7) / 8, dg.n_views);
        k_count_views<N><<<grid, 128, 0, st>>>(dg, count, qr);
    }
    return launch_status("count launch");
}

// c: coefficient array (never empty); y: projection array (may be empty, and
// then NULL)
static spl_status check_call(const spl_geometry *g, const spl_basis_desc *b, const void *c, const void *y)
{
    clear_error();
    if (!g) return fail(SPL_ERR_ARG, "geometry is NULL");
    spl_status s = check_basis(b);
    if (s != SPL_OK) return s;
    if (!c) return fail(SPL_ERR_ARG, "coefficient pointer is NULL");
    if (!y && g->dev.n_rays > 0) return fail(SPL_ERR_ARG, "projection pointer is NULL");
    if (b->mode == SPL_FP_MLP) {
        if (spl_mlp_degree(b->mlp) != b->degree)
            return fail(SPL_ERR_ARG, "MLP degree %d does not match basis degree %d", spl_mlp_degree(b->mlp), b->degree);
        if (g->dev.kind == SPL_RAYS) return fail(SPL_ERR_UNSUPPORTED, "MLP footprint needs a view geometry");
    }
    return SPL_OK;
}

#define SPL_DISPATCH(deg, fn, ...)                                                                                   \
    switch (deg) {                                                                                                   \
    case 0: return fn<0>(__VA_ARGS__);                                                                               \
    case 1: return fn<1>(__VA_ARGS__);                                                                               \
    case 2: return fn<2>(__VA_ARGS__);                                                                               \
    default: return fn<3>(__VA_ARGS__);                                                                              \
    }

extern "C" spl_status spl_forward(const spl_geometry *g, const spl_basis_desc *b, const float *c_dev, float *y_dev,
                                  void *stream)
{
    spl_status s = check_call(g, b, c_dev, y_dev);
    if (s != SPL_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    if (b->mode == SPL_FP_MLP) return spl::forward_mlp(g, b, c_dev, y_dev, st);
    if (b->mode == SPL_FP_TABLE) return spl::table_forward(g, b, c_dev, y_dev, st);
    SPL_DISPATCH(b->degree, forward_quad, g, b, c_dev, y_dev, st)
}

extern "C" spl_status spl_adjoint(const spl_geometry *g, const spl_basis_desc *b, const float *y_dev, float *c_dev,
                                  void *stream)
{
    spl_status s = check_call(g, b, c_dev, y_dev);
    if (s != SPL_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    if (b->mode == SPL_FP_MLP) return spl::adjoint_mlp(g, b, y_dev, c_dev, st);
    if (b->mode == SPL_FP_TABLE) return spl::table_adjoint(g, b, y_dev, c_dev, st);
    if (b->adjoint != SPL_ADJ_AUTO && b->adjoint != SPL_ADJ_GATHER && b->adjoint != SPL_ADJ_SCATTER)
        return fail(SPL_ERR_ARG, "unknown adjoint form %d", b->adjoint);
    SPL_DISPATCH(b->degree, adjoint_quad, g, b, y_dev, c_dev, st)
}

extern "C" spl_status spl_count_pairs(const spl_geometry *g, int degree, unsigned long long *count_dev, void *stream)
{
    clear_error();
    if (!g || !count_dev) return fail(SPL_ERR_ARG, "NULL argument");
    if (degree < 0 || degree > 3) return fail(SPL_ERR_ARG, "degree %d not in 0..3", degree);
    SPL_DISPATCH(degree, count_pairs, g, count_dev, (cudaStream_t)stream)
}
