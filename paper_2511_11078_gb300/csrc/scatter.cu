// scatter.cu -- the adjoint A^T (Sec. 2.3) as a ray-driven scatter, degrees
// 1 to 3: explicit rays, cone views and the parallel views outside the flat
// class.
//
// One thread per ray walks the pieces of the piece march (spl_march.cuh) with
// the (n+1)^3 register window of footprint integrals; the face that leaves
// the window at an event is reduced into the target with vector atomics.
//
// Target: three layouts of c, one per contiguous axis b (the ray's smallest
// direction component), each kept as copies shifted by 0 .. 3 floats, so
// that a row of n+1 values along b is one aligned 16-byte reduction (8 bytes
// for n = 1) into the copy in which it starts a group.  Every axis is padded
// on both sides, so no entry of a face needs a bounds test, and rows are
// a multiple of 4 floats apart, so the copy is chosen once per b crossing and
// not once per row.  k_fold_* add the layouts into c (or the FP64 total of the
// batches) and leave them cleared for the next call.  Explicit rays that do not
// lie side by side take fewer copies, or single values into one layout
// (scatter_form).
//
// The march keeps, next to its 64 accumulators, only what every piece needs
// in registers (4 blocks of 128 threads per SM); the ray's constants sit in
// shared memory.  Positions are 64-bit fixed point (spl_line.cuh), one add per
// cell and axis.  Bound by issue and the FMA pipe together (60 and 62 % busy
// on 8 views of the 256^3 cone, the L2's tag lookups at 66 %) and by those tag
// lookups on the 512^3 helical views (86 %).  Against
// the mirrored march with bounds tests and double-float positions at 3 blocks
// per SM: 8 such views 9.5 -> 7.35 ms, 8 helical views of 512^3 71.2 -> 54.9, 64
// general parallel views of 128^3 8.4 -> 6.0, quadratic 180 x 180 x 50 8.5 ->
// 5.3 (rows of three were scalar atomics), 24^3 0.18 -> 0.08.  Measured and not
// kept: b events in a branch of their own, which leaves one select per entry
// instead of two (the register allocation spills: 7.3 -> 9.5 ms); 3 blocks per
// SM (7.3 -> 7.8).
#include <math.h>

#include <new>

#include "spl_host.h"
#include "spl_line.cuh"

namespace spl {

// every axis is padded by 3 on both sides, whatever the degree, so that the
// degrees share the layouts' cleared state
constexpr int kPad = 3;
template <int N> constexpr int kCopies = N == 0 ? 1 : (N == 1 ? 2 : 4);

struct ScatterTarget {
    float *lay[3];  // contiguous axis x, y, z; NULL where no ray has it as b axis
    size_t cs;      // copy stride in floats, a multiple of 4
    int one;        // the layout of every ray (form 0), or -1: that of its b axis
};

// Layout with contiguous axis b: rows of `row` floats (room for the shift and
// for the fourth value of a quadratic row), `slab` floats per step of the
// higher of the other two axes.
struct ScatterDims {
    int row, slab;
    long long total;
};
__host__ __device__ inline ScatterDims scatter_dims(const int (&n)[3], int b)
{
    ScatterDims D;
    D.row = (sel3(b, n[0], n[1], n[2]) + 2 * kPad + 4 + 3) & ~3;
    D.slab = D.row * ((b == 0 ? n[1] : n[0]) + 2 * kPad);
    D.total = (long long)D.slab * ((b == 2 ? n[1] : n[2]) + 2 * kPad);
    return D;
}

// ---------------------------------------------------------------- ray set-up
struct __align__(16) ScatterRay {
    long long A, B;    // v_a, v_b at the start of cell c
    long long RA, RB;  // and their steps, >= 0
    float ia, ib;      // reciprocals of ra, rb
    float ra, rb;      // steps per cell, 0 <= rb <= ra <= 1
    float yv;          // y / |w_d|
    int four;          // cubic: every piece takes four Gauss nodes (line_four)
    int lim_a, lim_b;  // the window meets the grid while 0 <= Q < lim
    int c, cl;         // first and last cell (none: c > cl)
    int sd, sa;        // signed strides of d and a in the target
    float *base;       // target of window entry (0, 0, 0) at cell c, QA = QB = 0, in copy 0
    int sb, pad;       // stride of b in the target
};

// The line {s + t w}, oriented so that its b component is >= 0 and mirrored
// along d and a where their components are negative (beta is even), so every
// coordinate grows along the ray.  R comes with an empty cell range and
// keeps it when the line meets no support.
template <int N>
__device__ __forceinline__ void scatter_setup(const DevGeom &g, const ScatterTarget &T, const double (&s)[3],
                                              const double (&w)[3], float y, ScatterRay &R)
{
    constexpr double W = 0.5 * (N + 1);
    const double m0 = fabs(w[0]), m1 = fabs(w[1]), m2 = fabs(w[2]);
    int d = 0;
    if (m1 > m0) d = 1;
    if (m2 > (d == 1 ? m1 : m0)) d = 2;
    int a = d == 0 ? 1 : 0, b = d == 2 ? 1 : 2;
    if (sel3(b, m0, m1, m2) > sel3(a, m0, m1, m2)) {
        const int t = a;
        a = b;
        b = t;
    }
    const double wd = sel3(d, w[0], w[1], w[2]), wa = sel3(a, w[0], w[1], w[2]), wb = sel3(b, w[0], w[1], w[2]);
    const int nd = sel3(d, g.n[0], g.n[1], g.n[2]), na = sel3(a, g.n[0], g.n[1], g.n[2]),
              nb = sel3(b, g.n[0], g.n[1], g.n[2]);
    // (a zero component is not mirrored: the half-open box of degree 0 tells the sides apart)
    const bool flip = wb < 0.0, nd_ = (wd < 0.0) != flip, na_ = wa != 0.0 && (wa < 0.0) != flip;
    const double u0 = s[0] - g.org[0], u1 = s[1] - g.org[1], u2 = s[2] - g.org[2];
    double ud = sel3(d, u0, u1, u2), ua = sel3(a, u0, u1, u2);
    const double ub = sel3(b, u0, u1, u2);
    if (nd_) ud = (nd - 1) - ud;
    if (na_) ua = (na - 1) - ua;
    const double iw = 1.0 / fabs(wd);
    double ra = fabs(wa) * iw, rb = fabs(wb) * iw;
    if (ra < 1e-30) ra = 0.0;
    if (rb < 1e-30) rb = 0.0;
    const double q2 = fma(ra, ra, fma(rb, rb, 1.0));
    const float r0 = sqrtf((float)q2);
    // the three axes' weights come out 1.27e-7 too large together (spl_line.cuh)
    const float scale = r0 + fmaf(-weight_excess<N>(3), r0, (float)fma(-(double)r0, (double)r0, q2) * (0.5f / r0));
    R.yv = y * scale;
    R.ra = (float)ra;
    R.rb = (float)rb;
    R.ia = ra > 0.0 ? 1.0f / R.ra : 1.0f;
    R.ib = rb > 0.0 ? 1.0f / R.rb : 1.0f;
    if (N == 3) R.four = line_four(R.ra, R.rb);
    const double a0 = fma(-(W + ud), ra, ua) + W, b0 = fma(-(W + ud), rb, ub) + W;
    float vmin = 0.0f, vmax = (float)(nd + N);
    if (ra > 0.0) {
        vmin = fmaxf(vmin, (float)(0.0 - a0) * R.ia);
        vmax = fminf(vmax, (float)((double)(na + N) - a0) * R.ia);
    } else if (!(a0 >= 0.0 && a0 < (double)(na + N))) {
        return;
    }
    if (rb > 0.0) {
        vmin = fmaxf(vmin, (float)(0.0 - b0) * R.ib);
        vmax = fminf(vmax, (float)((double)(nb + N) - b0) * R.ib);
    } else if (!(b0 >= 0.0 && b0 < (double)(nb + N))) {
        return;
    }
    if (!(vmax >= vmin - 1.0f)) return;
    // one cell of margin on both ends: the ray has left the grid's supports
    // at the end of the last cell
    const int c = max((int)floorf(vmin) - 1, 0);
    R.c = c;
    R.cl = min((int)floorf(vmax) + 1, nd + N - 1);
    constexpr double kOne = (double)(1LL << kLineFrac);
    R.RA = __double2ll_rn(ra * kOne);
    R.RB = __double2ll_rn(rb * kOne);
    R.A = __double2ll_rn(fma((double)c, ra, a0) * kOne);
    R.B = __double2ll_rn(fma((double)c, rb, b0) * kOne);
    R.lim_a = na + N;
    R.lim_b = nb + N;
    // strides of the layout with contiguous axis e: rows, then slabs
    const int e = T.one >= 0 ? T.one : b;
    const ScatterDims D = scatter_dims(g.n, e);
    auto stride = [&](int x) { return x == e ? 1 : (x == (e == 2 ? 1 : 2) ? D.slab : D.row); };
    const int st_d = stride(d), st_a = stride(a);
    R.sd = nd_ ? -st_d : st_d;
    R.sa = na_ ? -st_a : st_a;
    R.sb = stride(b);
    // window entry (0, 0, 0) is basis (c - N, QA - N, QB - N); basis l sits at
    // l + kPad, a mirrored one at n - 1 - l + kPad
    const long long od = nd_ ? nd - 1 - (c - N) + kPad : c - N + kPad, oa = na_ ? na - 1 + N + kPad : kPad - N;
    float *lay = sel3(e, T.lay[0], T.lay[1], T.lay[2]);
    if (!lay) {  // an axis that scatter_axes ruled out (not expected)
        atomicOr(g.err, 1);
        R.cl = c - 1;
        return;
    }
    R.base = lay + (od * st_d + oa * st_a + (long long)(kPad - N) * R.sb);
}

// ---------------------------------------------------------------- the march
// Reductions without a result into the target, spelled out: its address comes
// from shared memory, so the compiler cannot see that it is global and an
// atomicAdd becomes an atomic with a result that the warp waits for (8 cone
// views 9.4 ms against 6.0).
__device__ __forceinline__ void red1(float *p, float v)
{
    asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "f"(v) : "memory");
}
__device__ __forceinline__ void red2(float *p, float v0, float v1)
{
    asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};" ::"l"(__cvta_generic_to_global(p)), "f"(v0), "f"(v1)
                 : "memory");
}
// A row of N + 1 values along b, which starts on a boundary of CP floats;
// CP = 0: values sb floats apart.
template <int N, int CP>
__device__ __forceinline__ void row_add(float *p, const float (&v)[N + 1], int sb)
{
    if constexpr (CP == 4)
        asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(__cvta_generic_to_global(p)),
                     "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(N == 3 ? v[N] : 0.0f)
                     : "memory");
    else {
        constexpr int P = CP == 2 ? (N + 1) / 2 : 0;
#pragma unroll
        for (int k = 0; k < P; ++k) red2(p + 2 * k, v[2 * k], v[2 * k + 1]);
#pragma unroll
        for (int k = 2 * P; k <= N; ++k) red1(p + (CP == 0 ? (long long)k * sb : k), v[k]);
    }
}

// March over part `seg` of 2^ls equal parts of the ray's cells.  Returns
// false if the event bound was reached.  HOME: the single values of a b event,
// which need no alignment, go to copy 0 and not to the ray's current copy
// (ScatterScratch::home).
template <int N, int CP, bool HOME>
__device__ __forceinline__ bool scatter_march(const ScatterRay &R, int seg, int ls, size_t cs, const QuadRule &qr)
{
    constexpr int M = GL<N>::M, C1 = CP > 0 ? CP : 1;
    const int sb = CP > 0 ? 1 : R.sb;
    const int cells = R.cl - R.c + 1, k0 = (int)(((long long)cells * seg) >> ls),
              k1 = (int)(((long long)cells * (seg + 1)) >> ls);
    const bool four = N == 3 && __all_sync(0xffffffffu, k0 >= k1 || R.four);
    if (k0 >= k1) return true;
    int left = k1 - k0;
    long long A = R.A + R.RA * k0, B = R.B + R.RB * k0;
    int QA = (int)(A >> kLineFrac), QB = (int)(B >> kLineFrac);
    const float ra = R.ra, rb = R.rb;
    // target of window entry (0, 0, 0), at float lo = QB + kPad - N of its
    // row: copy j = -lo mod C1 holds it at lo + j, where a group starts
    constexpr int kLo = kPad - N;
    float *wp;
    {
        const int j = -(QB + kLo) & (C1 - 1);
        wp = R.base + (long long)k0 * R.sd + (long long)QA * R.sa + ((long long)QB * sb + j) + (long long)((size_t)j * cs);
    }
    float acc[N + 1][N + 1][N + 1];
#pragma unroll
    for (int d = 0; d <= N; ++d)
#pragma unroll
        for (int i = 0; i <= N; ++i)
#pragma unroll
            for (int k = 0; k <= N; ++k) acc[d][i][k] = 0.0f;
    float ga, gb, ta, tb, t0;
    // fractions at the cell's start and the crossings inside it (2: none);
    // whether there is one is decided by the integers, so the window's frame
    // and the cell's agree everywhere on the ray
    auto cell = [&]() {
        constexpr float kUnit = 1.0f / 4294967296.0f;
        const uint4 r = lds128(&R.RA), e = lds128(&R.ia);
        ga = __uint2float_rn((unsigned)(A >> (kLineFrac - 32))) * kUnit;
        gb = __uint2float_rn((unsigned)(B >> (kLineFrac - 32))) * kUnit;
        const long long An = A + (long long)(((unsigned long long)r.y << 32) | r.x);
        const long long Bn = B + (long long)(((unsigned long long)r.w << 32) | r.z);
        ta = (int)(An >> kLineFrac) != QA ? fminf((1.0f - ga) * __uint_as_float(e.x), 1.0f) : 2.0f;
        tb = (int)(Bn >> kLineFrac) != QB ? fminf((1.0f - gb) * __uint_as_float(e.y), 1.0f) : 2.0f;
        A = An;  // the next cell's start
        B = Bn;
        t0 = 0.0f;
    };
    cell();
    int ev = 0;
#pragma unroll 1
    while (true) {
        const uint4 yl = lds128(&R.yv);
        const bool in = (unsigned)QA < yl.z && (unsigned)QB < yl.w;
        const float t1 = fminf(fminf(ta, tb), 1.0f);
        if (t1 > t0 && in) {
            const float half = 0.5f * (t1 - t0), mid = 0.5f * (t0 + t1), hs = half * __uint_as_float(yl.x);
            auto node = [&](float x, float wt) {
                const float t = fmaf(half, x, mid);
                float wd[N + 1], wa[N + 1], wb[N + 1];
                bweights<N>(t, wd);
                bweights<N>(fmaf(ra, t, ga), wa);
                bweights<N>(fmaf(rb, t, gb), wb);
                window_update<N>(acc, wd, wa, wb, hs * wt);
            };
            if constexpr (N == 3) {
                if (four) {
#pragma unroll
                    for (int q = 0; q < M - 1; ++q) node(qr.x1[q], qr.w1[q]);
                } else {
#pragma unroll
                    for (int q = 0; q < M; ++q) node(qr.x[q], qr.w[q]);
                }
            } else {
#pragma unroll
                for (int q = 0; q < M; ++q) node(qr.x[q], qr.w[q]);
            }
        }
        t0 = fmaxf(t0, t1);
        if (++ev > qr.cap) return false;
        const bool evA = ta <= tb && ta <= 1.0f, evB = !evA && tb <= 1.0f, evD = !evA && !evB;
        const int2 st = make_int2(R.sd, R.sa);
        // the face that leaves: D: (0, x, .), A: (x, 0, .): rows along b;
        // B: (x, y, 0): single values
        if (in) {
            if (evB) {
                float *w0 = HOME ? wp - (-(QB + kLo) & (C1 - 1)) * (long long)(cs + 1) : wp;
#pragma unroll
                for (int x = 0; x <= N; ++x)
#pragma unroll
                    for (int y = 0; y <= N; ++y) red1(w0 + ((long long)x * st.x + (long long)y * st.y), acc[x][y][0]);
            } else {
                const long long sx = evD ? st.y : st.x;
#pragma unroll
                for (int x = 0; x <= N; ++x) {
                    float v[N + 1];
#pragma unroll
                    for (int k = 0; k <= N; ++k) v[k] = evD ? acc[0][x][k] : acc[x][0][k];
                    row_add<N, CP>(wp + x * sx, v, sb);
                }
            }
        }
        // shift along the event's axis (in place: reads only higher indices)
#pragma unroll
        for (int d = 0; d <= N; ++d)
#pragma unroll
            for (int i = 0; i <= N; ++i)
#pragma unroll
                for (int k = 0; k <= N; ++k) {
                    const float nd = d < N ? acc[(d < N ? d + 1 : d)][i][k] : 0.0f;
                    const float na = i < N ? acc[d][(i < N ? i + 1 : i)][k] : 0.0f;
                    const float nb = k < N ? acc[d][i][(k < N ? k + 1 : k)] : 0.0f;
                    acc[d][i][k] = evD ? nd : (evA ? na : nb);
                }
        if (evD) {
            if (--left == 0) break;
            wp += st.x;
            cell();
            ev = 0;
        } else if (evA) {
            ++QA;
            ga -= 1.0f;
            ta = 2.0f;
            wp += st.y;
        } else {
            // the row start moves on by one: the copy before holds it at the
            // same position, copy 0's successor is copy C1 - 1, C1 further on
            const bool last = ((QB + kLo) & (C1 - 1)) == 0;
            ++QB;
            gb -= 1.0f;
            tb = 2.0f;
            wp += last ? (long long)((C1 - 1) * cs) + C1 * sb : -(long long)cs;
        }
    }
    // what the window still holds (it is shifted: layers c + 1 - N ..), for a
    // part of a ray that ends inside the grid
    const bool in = (unsigned)QA < (unsigned)R.lim_a && (unsigned)QB < (unsigned)R.lim_b;
    if (in) {
        wp += R.sd;
#pragma unroll
        for (int d = 0; d < N; ++d)
#pragma unroll
            for (int i = 0; i <= N; ++i) row_add<N, CP>(wp + ((long long)d * R.sd + (long long)i * R.sa), acc[d][i], sb);
    }
    return true;
}

// ---------------------------------------------------------------- kernels
template <int N> struct ScatterBlocks { static constexpr int value = N == 3 ? 4 : (N == 2 ? 5 : 8); };

// rays r0 .. r1 - 1, 2^ls threads each
template <int N, int CP, bool HOME>
__global__ void __launch_bounds__(128, ScatterBlocks<N>::value)
    k_scatter_rays(DevGeom g, ScatterTarget T, const float *__restrict__ y, QuadRule qr, long long r0, long long r1, int ls)
{
    __shared__ ScatterRay rays[128];
    const int t = threadIdx.x;
    const long long rb = r0 + (((long long)blockIdx.x * 128) >> ls);
    if (t < (128 >> ls)) {
        rays[t].c = 0;
        rays[t].cl = -1;
        if (rb + t < r1) {
            const float yr = __ldg(y + rb + t);
            if (yr != 0.0f) {
                double s[3], w[3];
                explicit_ray(g, rb + t, s, w);
                scatter_setup<N>(g, T, s, w, yr, rays[t]);
            }
        }
    }
    __syncthreads();
    if (!scatter_march<N, CP, HOME>(rays[t >> ls], t & ((1 << ls) - 1), ls, T.cs, qr)) atomicOr(g.err, 1);
}

// Whether a warp's eight consecutive lanes run along detector v: along the
// axis that moves more along the rays' b axis, so that the lanes' rows share
// 128-byte lines (64 general parallel views 6.10 ms, 6.54 the other way; cone
// views alike).  Decided for the view's central ray.
__device__ __forceinline__ bool scatter_lanes_along_v(const DevGeom &g, int k)
{
    const ViewPose &P = g.views[k];
    float w[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) w[e] = fabsf((float)(g.kind == SPL_PARALLEL ? P.src[e] : P.dc[e] - P.src[e]));
    const int b = w[0] < w[1] ? (w[2] < w[0] ? 2 : 0) : (w[2] < w[1] ? 2 : 1);
    return fabs(sel3(b, P.dv[0], P.dv[1], P.dv[2])) >= fabs(sel3(b, P.du[0], P.du[1], P.du[2]));
}

// views v0 + blockIdx.z (of order[], when given); the block's pixels form the
// tiles of line_tile
template <int N, bool HOME>
__global__ void __launch_bounds__(128, ScatterBlocks<N>::value)
    k_scatter_views(DevGeom g, ScatterTarget T, const float *__restrict__ y, QuadRule qr, const int *order, int v0, int ls)
{
    __shared__ ScatterRay rays[128];
    const int t = threadIdx.x;
    const int k = order ? order[v0 + blockIdx.z] : v0 + (int)blockIdx.z;
    if (t < (128 >> ls)) {
        rays[t].c = 0;
        rays[t].cl = -1;
        int iu, iv;
        line_tile(t, ls, scatter_lanes_along_v(g, k), iu, iv);
        if (iu < g.nu && iv < g.nv) {
            const float yr = __ldg(y + ((long long)k * g.nv + iv) * g.nu + iu);
            if (yr != 0.0f) {
                double s[3], w[3];
                line_pixel(g, k, iu, iv, s, w);
                scatter_setup<N>(g, T, s, w, yr, rays[t]);
            }
        }
    }
    __syncthreads();
    if (!scatter_march<N, kCopies<N>, HOME>(rays[t >> ls], t & ((1 << ls) - 1), ls, T.cs, qr)) atomicOr(g.err, 1);
}

// ---------------------------------------------------------------- fold
// out = src + sum over the layouts and their copies, and the layouts cleared
// for the next call.  HBM-bound: 16 bytes read and 16 cleared per coefficient
// and layout.  A layout at a time through 32 x 32 tiles, both sides coalesced,
// all copies of a thread's four coefficients in flight before any is cleared
// (a single kernel over all three layouts in 32 x 16 x 16 tiles took 14 ms at
// 512^3, these 4); small grids, which sit in the L2 and where a launch counts,
// one thread per coefficient and all layouts in one launch (k_fold_small).
//
// What a fold starts from and where it ends:
enum { FOLD_ZERO = 0, FOLD_C = 1 };                              // base: nothing, what c holds
enum { FOLD_TO_C = 0, FOLD_TO_ACC = 1, FOLD_ADD_ACC = 2, FOLD_ACC_TO_C = 3 };  // acc: the FP64 total

struct FoldOut {
    int base, fin;
    float *c;
    double *acc;
    // what the outcome adds to the layouts' sum at o; read before anything is
    // written (a read between the writes waits for each of them in turn)
    __device__ __forceinline__ float from_c(long long o) const { return base == FOLD_C ? c[o] : 0.0f; }
    __device__ __forceinline__ double from_acc(long long o) const { return fin >= FOLD_ADD_ACC ? acc[o] : 0.0; }
    __device__ __forceinline__ void put(long long o, float v, double a) const
    {
        if (fin == FOLD_TO_C) c[o] = v;
        else if (fin == FOLD_ACC_TO_C) c[o] = (float)(a + (double)v);
        else acc[o] = a + (double)v;
    }
};

template <int CP> __device__ __forceinline__ float fold_sum(const float (&v)[CP])
{
    if constexpr (CP == 1) return v[0];
    else if constexpr (CP == 2) return v[0] + v[1];
    else return (v[0] + v[1]) + (v[2] + v[3]);
}

// One layout, contiguous axis B: block (b tile, row tile, slab); rows are y
// at z = slab (B = x), x at z = slab (B = y), x at y = slab (B = z)
template <int CP, int B>
__global__ void __launch_bounds__(256) k_fold_layout(int3 n, float *lay, size_t cs, FoldOut out)
{
    __shared__ float tile[32][33];
    const int dims[3] = {n.x, n.y, n.z};
    const ScatterDims D = scatter_dims(dims, B);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, sl = blockIdx.z;
    const int b0 = blockIdx.x * 32, r0 = blockIdx.y * 32, nb = B == 0 ? n.x : (B == 1 ? n.y : n.z), nr = B == 0 ? n.y : n.x;
    float v[4][CP], vc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    double va[4] = {0.0, 0.0, 0.0, 0.0};
    long long p[4], o[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int k = ty + 8 * u;
        p[u] = r0 + k < nr && b0 + tx < nb
                   ? (long long)(sl + kPad) * D.slab + (long long)(r0 + k + kPad) * D.row + (b0 + tx + kPad)
                   : -1;
        // this thread's outputs: along x, row k of the turned tile
        if (B == 0) o[u] = p[u] < 0 ? -1 : ((long long)sl * n.y + (r0 + k)) * n.x + (b0 + tx);
        else
            o[u] = b0 + k < nb && r0 + tx < n.x
                       ? (B == 1 ? (long long)sl * n.y + (b0 + k) : (long long)(b0 + k) * n.y + sl) * n.x + (r0 + tx)
                       : -1;
    }
    // all reads before any write, and no branch between them (outside the
    // grid: the first element, unused)
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int j = 0; j < CP; ++j) v[u][j] = lay[(p[u] < 0 ? 0 : p[u]) + (long long)(j * cs) + j];
    if (out.base == FOLD_C) {
#pragma unroll
        for (int u = 0; u < 4; ++u) vc[u] = out.c[o[u] < 0 ? 0 : o[u]];
    }
    if (out.fin >= FOLD_ADD_ACC) {
#pragma unroll
        for (int u = 0; u < 4; ++u) va[u] = out.acc[o[u] < 0 ? 0 : o[u]];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const float t = fold_sum<CP>(v[u]);
        if (B == 0) vc[u] += t;
        else tile[ty + 8 * u][tx] = t;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (p[u] < 0) continue;
#pragma unroll
        for (int j = 0; j < CP; ++j) lay[p[u] + (long long)(j * cs) + j] = 0.0f;
    }
    if (B != 0) __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u)
        if (o[u] >= 0) out.put(o[u], B == 0 ? vc[u] : vc[u] + tile[tx][ty + 8 * u], va[u]);
}

template <int CP>
__global__ void __launch_bounds__(128) k_fold_small(int3 n, ScatterTarget T, FoldOut out)
{
    const int i = blockIdx.x * 128 + threadIdx.x;
    if (i >= n.x * n.y * n.z) return;
    const int x = i % n.x, y = i / n.x % n.y, z = i / (n.x * n.y);
    const int dims[3] = {n.x, n.y, n.z};
    const float vc = out.from_c(i);
    const double va = out.from_acc(i);
    float v[3][CP];
    float *p[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const ScatterDims D = scatter_dims(dims, b);
        const int lo = b == 0 ? x : (b == 1 ? y : z), row = b == 0 ? y : x, slab = b == 2 ? y : z;
        p[b] = T.lay[b] ? T.lay[b] + (long long)(slab + kPad) * D.slab + (long long)(row + kPad) * D.row + (lo + kPad) : nullptr;
#pragma unroll
        for (int j = 0; j < CP; ++j) v[b][j] = p[b] ? p[b][(long long)(j * T.cs) + j] : 0.0f;
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (!p[b]) continue;
#pragma unroll
        for (int j = 0; j < CP; ++j) p[b][(long long)(j * T.cs) + j] = 0.0f;
    }
    out.put(i, vc + ((fold_sum<CP>(v[0]) + fold_sum<CP>(v[1])) + fold_sum<CP>(v[2])), va);
}

// ---------------------------------------------------------------- host side
struct ScatterScratch {
    ScatterTarget T;
    void *block;
    size_t bytes;
    int form[4];     // per degree (scatter_form)
    int batches[4];  // per degree (scatter_batches)
    // per degree: single values go to copy 0.  Where the copies outgrow the L2,
    // that makes the target smaller (8 helical views 55.5 -> 54.9 ms); otherwise
    // many rays through a small grid would meet at one address (300 000 through
    // 12^3: 0.53 ms, 0.39 in the rays' copies).  Linear splines: always (64
    // general parallel views of 128^3 1.61 -> 1.53 ms).
    bool home[4];
    bool dirty;      // to be cleared before the next call: new, or a launch failed between scatter and fold
};

// Axes that can be the smallest component of a line of the geometry (a
// superset).
static unsigned scatter_axes(const spl_geometry *g, const double *ray_dirs)
{
    unsigned mask = 0;
    line_bounds(g, ray_dirs, [&](const double (&lo)[3], const double (&hi)[3]) {
        for (int e = 0; e < 3; ++e) {
            bool can = true;
            for (int f = 0; f < 3; ++f) can = can && lo[e] <= hi[f] * (1.0 + 1e-9);
            if (can) mask |= 1u << e;
        }
        return mask != 7u;
    });
    return mask;
}

// Whether explicit rays are scattered: of 4096 pairs of neighbours in the
// caller's order, half or more lie more than a sixteenth of the grid apart
// (at the points nearest the grid's centre, or by their directions half a
// grid away from it), so that the rays a GPU works on at a time reach all over
// the grid.
static bool scattered_rays(const DevGeom &g, const double *dirs, const double *points)
{
    const long long pairs = g.n_rays - 1, step = pairs / 4096 > 1 ? pairs / 4096 : 1;
    const int n = g.n[0] > g.n[1] ? (g.n[0] > g.n[2] ? g.n[0] : g.n[2]) : (g.n[1] > g.n[2] ? g.n[1] : g.n[2]);
    long long seen = 0, apart = 0;
    for (long long r = 0; r < pairs; r += step) {
        double w[2][3], p[2][3];
        for (int i = 0; i < 2; ++i) {
            const double *d = dirs + 3 * (r + i), *s = points + 3 * (r + i);
            const double l = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
            double t = 0.0;
            for (int e = 0; e < 3; ++e) {
                w[i][e] = d[e] / l;
                p[i][e] = s[e] - (g.org[e] + 0.5 * (g.n[e] - 1));
                t += p[i][e] * w[i][e];
            }
            for (int e = 0; e < 3; ++e) p[i][e] -= t * w[i][e];
        }
        // (a line has two directions)
        const double sg = w[0][0] * w[1][0] + w[0][1] * w[1][1] + w[0][2] * w[1][2] < 0.0 ? -1.0 : 1.0;
        double dp = 0.0, dw = 0.0;
        for (int e = 0; e < 3; ++e) {
            dp += (p[0][e] - p[1][e]) * (p[0][e] - p[1][e]);
            dw += (w[0][e] - sg * w[1][e]) * (w[0][e] - sg * w[1][e]);
        }
        ++seen;
        apart += sqrt(dp) + 0.5 * n * sqrt(dw) > n / 16.0 ? 1 : 0;
    }
    return 2 * apart > seen;
}

// Form of a degree's reductions: the number of shifted copies, or 0 for single
// values into one layout.  Rays side by side keep working on one part of the
// grid, and a row in one reduction (kCopies) is the fewest of them.  Scattered
// rays reach the whole target all the time, and it has to stay in the L2: the
// most copies with which the layouts do, and one layout (4 bytes a
// coefficient, a twelfth of the most) where they do not with two.  300 000
// random rays, ms with 4 copies, 2 copies, one layout (the L2 holds 135 MB):
//   cubic      128^3   2.55   2.74     -     115 MB in 4 copies
//              144^3   5.28   3.16    5.14    81 MB in 2
//              192^3  12.5    9.38    6.49   183 MB in 2
//              256^3  22.2   19.6     8.65
//              400^3  40.9   39.9    30.1
//   linear     160^3          1.14    1.51   109 MB in 2
//              192^3          3.28    1.71   183 MB in 2
//              400^3         15.8     9.13
// (single values into the three layouts of one copy: cubic 192^3 6.57, 256^3
// 16.9, 400^3 46.5; four copies of the one layout by ray, cubic 192^3 600 000
// rays 14.7 against 14.5, linear 3.98 against 3.53).
static int scatter_form(const DevGeom &g, unsigned mask, bool scattered, int degree)
{
    const int most = degree == 0 ? kCopies<0> : (degree == 1 ? kCopies<1> : kCopies<3>);
    if (!scattered) return most;
    size_t one = 0;  // bytes of the layouts with one copy
    for (int b = 0; b < 3; ++b) one += ((mask >> b) & 1u) ? scatter_dims(g.n, b).total * sizeof(float) : 0;
    for (int cp = most; cp >= (degree == 0 ? 1 : 2); cp /= 2)
        if (cp * one <= l2_bytes()) return cp;
    return 0;
}

// Into how many batches the rays of a call are divided where the form has
// fewer copies than kCopies.  A running FP32 sum of T terms of random sign
// rounds T / 2 times the square of one rounding of its size; p partial sums
// (layouts times copies) round T / (2 p), and `tree` more where they are added
// up.  With the FP64 total of the batches, (T / p) / (T / p0 + 2 (tree0 -
// tree)) of them round as much as kCopies copies (p0, tree0).  A^T of random
// rays, relative error against FP64 with 4 copies, in one batch, and so
// divided: cubic 192^3, 300 000 rays 1.47e-7, 2.81e-7, 1.46e-7; 60 000 rays
// 1.29e-7, 1.63e-7, 1.30e-7.
static double scatter_tree(int copies, int layouts)
{
    return (copies >= 4 ? 2.0 : (copies == 2 ? 1.0 : 0.0)) + (layouts == 3 ? 1.7 : (layouts == 2 ? 1.0 : 0.0));
}
static int scatter_batches(const DevGeom &g, unsigned mask, int degree, int form)
{
    const int most = degree == 0 ? kCopies<0> : (degree == 1 ? kCopies<1> : kCopies<3>);
    if (form == most) return 1;
    int layouts = 0;
    for (int b = 0; b < 3; ++b) layouts += (mask >> b) & 1u;
    const double n = (g.n[0] + g.n[1] + g.n[2]) / 3.0, nc = (double)g.n[0] * g.n[1] * g.n[2];
    // a ray crosses about 1.5 n cells with (degree + 1)^2 new bases each
    const double T = g.n_rays * 1.5 * n * (degree + 1) * (degree + 1) / nc;
    const double p = form == 0 ? 1 : layouts * form, tree = form == 0 ? 0.0 : scatter_tree(form, layouts);
    const double k = (T / p) / (T / (layouts * most) + 2.0 * (scatter_tree(most, layouts) - tree));
    return T > 1.0 && k > 1.0 ? (int)ceil(k) : 1;
}

spl_status scatter_create(spl_geometry *g, const double *ray_dirs, const double *ray_points)
{
    const DevGeom &dg = g->dev;
    g->scatter = nullptr;
    g->scattered = dg.kind == SPL_RAYS && dg.n_rays > 0 && scattered_rays(dg, ray_dirs, ray_points);
    if (dg.n_rays == 0 || (dg.kind == SPL_PARALLEL && dg.n_flat == dg.n_views)) return SPL_OK;
    const unsigned mask = scatter_axes(g, ray_dirs);
    ScatterScratch *S = new (std::nothrow) ScatterScratch();
    if (!S) return fail(SPL_ERR_OOM, "host allocation failed");
    // copies of each layout that some degree takes; the first one also serves form 0
    const int first = (mask & 1u) ? 0 : ((mask & 2u) ? 1 : 2);
    int copies = 0;
    for (int n = 0; n < 4; ++n) {
        S->form[n] = scatter_form(dg, mask, g->scattered, n);
        S->batches[n] = scatter_batches(dg, mask, n, S->form[n]);
        size_t bytes = 0;
        for (int b = 0; b < 3; ++b)
            bytes += ((mask >> b) & 1u) ? scatter_dims(dg.n, b).total * sizeof(float) * S->form[n] : 0;
        S->home[n] = n == 1 || bytes > l2_bytes();
        copies = S->form[n] > copies ? S->form[n] : copies;
    }
    size_t cs = 0, floats = 0, off[3];
    for (int b = 0; b < 3; ++b) {
        const size_t t = (size_t)scatter_dims(dg.n, b).total;
        if (((mask >> b) & 1u) && (copies > 0 || b == first) && t > cs) cs = t;
    }
    cs = (cs + 63) & ~(size_t)63;
    for (int b = 0; b < 3; ++b) {
        off[b] = floats;
        if ((mask >> b) & 1u) floats += cs * (copies > 0 ? copies : (b == first ? 1 : 0));
    }
    S->bytes = floats * sizeof(float);
    if (cudaMalloc(&S->block, S->bytes) != cudaSuccess) {
        const size_t bytes = S->bytes;
        cudaGetLastError();
        delete S;
        return fail(SPL_ERR_OOM, "cudaMalloc of the adjoint's layout copies (%zu bytes) failed", bytes);
    }
    S->dirty = true;
    S->T.cs = cs;
    S->T.one = first;
    for (int b = 0; b < 3; ++b)
        S->T.lay[b] = ((mask >> b) & 1u) && (copies > 0 || b == first) ? (float *)S->block + off[b] : nullptr;
    g->scatter = S;
    return SPL_OK;
}

// The layouts that a call of this degree reduces into and folds.
static ScatterTarget scatter_target(const ScatterScratch &S, int degree)
{
    ScatterTarget T = S.T;
    if (S.form[degree] > 0) T.one = -1;
    else
        for (int b = 0; b < 3; ++b) T.lay[b] = b == T.one ? T.lay[b] : nullptr;
    return T;
}

long long scatter_batch(const spl_geometry *g, int degree)
{
    const long long k = g->scatter->batches[degree];
    return (g->dev.n_rays + k - 1) / k;
}

bool scatter_in_batches(const spl_geometry *g)
{
    if (!g->scatter) return false;
    for (int n = 0; n < 4; ++n)
        if (g->scatter->batches[n] > 1) return true;
    return false;
}

void scatter_free(ScatterScratch *S)
{
    if (!S) return;
    cudaFree(S->block);
    delete S;
}

template <int N>
static spl_status scatter_n(const spl_geometry *g, const float *y, long long i0, long long i1, cudaStream_t st)
{
    const DevGeom &dg = g->dev;
    ScatterScratch &S = *g->scatter;
    const QuadRule qr = quad_rule(N);
    if (S.dirty) {
        const spl_status s = cuda_check(cudaMemsetAsync(S.block, 0, S.bytes, st), "adjoint layout clear");
        if (s != SPL_OK) return s;
        // (a captured clear only runs when its graph does)
        if (!stream_captures(st)) S.dirty = false;
    }
    if (dg.kind == SPL_RAYS) {
        const int form = S.form[N], ls = line_split(i1 - i0, ScatterBlocks<N>::value);
        const unsigned blocks = (unsigned)((((i1 - i0) << ls) + 127) / 128);
        const ScatterTarget T = scatter_target(S, N);
        auto launch = [&](auto kernel) { kernel<<<blocks, 128, 0, st>>>(dg, T, y, qr, i0, i1, ls); };
        if (form == 0) launch(k_scatter_rays<N, 0, false>);
        else if (N >= 2 && form == 2) launch(k_scatter_rays<N, N >= 2 ? 2 : kCopies<N>, false>);
        else if (S.home[N]) launch(k_scatter_rays<N, kCopies<N>, true>);
        else launch(k_scatter_rays<N, kCopies<N>, false>);
    } else {
        const int views = (int)(i1 - i0), ls = line_split((long long)views * dg.nu * dg.nv, ScatterBlocks<N>::value);
        auto launch = [&](auto kernel) {
            kernel<<<line_grid(dg, views, ls), 128, 0, st>>>(dg, scatter_target(S, N), y, qr,
                                                             dg.kind == SPL_PARALLEL ? dg.view_order : nullptr, (int)i0, ls);
        };
        if (S.home[N]) launch(k_scatter_views<N, true>);
        else launch(k_scatter_views<N, false>);
    }
    const spl_status s = cuda_check(cudaGetLastError(), "adjoint launch");
    if (s != SPL_OK) S.dirty = true;
    return s;
}

spl_status scatter_rays(const spl_geometry *g, int degree, const float *y, long long i0, long long i1, cudaStream_t st)
{
    switch (degree) {
    case 0: return scatter_n<0>(g, y, i0, i1, st);
    case 1: return scatter_n<1>(g, y, i0, i1, st);
    case 2: return scatter_n<2>(g, y, i0, i1, st);
    default: return scatter_n<3>(g, y, i0, i1, st);
    }
}

// Grids up to this many coefficients fold in one launch: 24^3 75 against 87 us
// an adjoint; 99 x 90 x 77 already takes longer that way (1.07 against 0.97
// ms), its y- and z-fast layouts being read across their rows.
constexpr long long kFoldSmall = 1LL << 18;

template <int CP>
static void launch_fold(const spl_geometry *g, const ScatterTarget &T, int base, int fin, float *c, cudaStream_t st)
{
    const DevGeom &dg = g->dev;
    const int3 n = make_int3(dg.n[0], dg.n[1], dg.n[2]);
    const long long nc = (long long)n.x * n.y * n.z;
    if (nc <= kFoldSmall) {
        k_fold_small<CP><<<(unsigned)((nc + 127) / 128), 128, 0, st>>>(n, T, FoldOut{base, fin, c, g->acc64});
        return;
    }
    // layout by layout through c, the last one to where the fold ends
    int last = 2;
    while (last > 0 && !T.lay[last]) --last;
    for (int b = 0; b <= last; ++b) {
        if (!T.lay[b]) continue;
        const FoldOut f{base, b == last ? fin : (int)FOLD_TO_C, c, g->acc64};
        auto grid = [](int nb, int nr, int ns) { return dim3((nb + 31) / 32, (nr + 31) / 32, ns); };
        if (b == 0) k_fold_layout<CP, 0><<<grid(n.x, n.y, n.z), 256, 0, st>>>(n, T.lay[0], T.cs, f);
        else if (b == 1) k_fold_layout<CP, 1><<<grid(n.y, n.x, n.z), 256, 0, st>>>(n, T.lay[1], T.cs, f);
        else k_fold_layout<CP, 2><<<grid(n.z, n.x, n.y), 256, 0, st>>>(n, T.lay[2], T.cs, f);
        base = FOLD_C;
    }
}

spl_status scatter_fold(const spl_geometry *g, int degree, int src, bool to64, float *c, cudaStream_t st)
{
    const int base = src == 1 ? FOLD_C : FOLD_ZERO;
    const int fin = to64 ? (src == 2 ? FOLD_ADD_ACC : FOLD_TO_ACC) : (src == 2 ? FOLD_ACC_TO_C : FOLD_TO_C);
    const ScatterTarget T = scatter_target(*g->scatter, degree);
    const int form = g->scatter->form[degree];
    if (form == 4) launch_fold<4>(g, T, base, fin, c, st);
    else if (form == 2) launch_fold<2>(g, T, base, fin, c, st);
    else launch_fold<1>(g, T, base, fin, c, st);
    const spl_status s = cuda_check(cudaGetLastError(), "adjoint fold launch");
    if (s != SPL_OK) g->scatter->dirty = true;
    return s;
}

}  // namespace spl
