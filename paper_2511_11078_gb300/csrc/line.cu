// line.cu -- forward projection A as line integrals of f itself (Eq. 2), on
// coefficients resampled once per call along the rays' dominant axis.
//
// f = sum_k c_k phi(x - k) is, on every cell [c, c+1) of axis d (v = u + W,
// the cells of the cell march), a polynomial in the position t in [0, 1] along
// d for each pair of transverse indices (la, lb).  With the cell's coefficients
// c_0 .. c_n along d and s = 1 - t it is
//   s (x + z g(s)) + t (y + w g(t)),
//   cubic:     x = c_1, y = c_2, z = (c_0 - 2 c_1 + c_2) / 6,
//              w = (c_1 - 2 c_2 + c_3) / 6, g(q) = q^2;
//   quadratic: x = y = c_1, z = (c_0 - c_1) / 2, w = (c_2 - c_1) / 2, g(q) = q;
//   linear:    x = c_0, y = c_1, z = w = 0.
// k_line_resample writes x, y, z, w of every cell and column as one float4
// (x, y as a float2 for n = 1; no y for n = 2).  A ray is cut into the pieces
// of the piece march (spl_march.cuh: cells along its dominant axis, split at
// the knot planes of the other two, r <= 1) and each piece is integrated with
// a Gauss-Legendre rule; a node needs two weight sets instead of three and
// contracts (n+1)^2 columns:
//   f(t) = (s, t) . sum_i wa_i sum_k wb_k ((x, y) + (g(s), g(t)) (z, w)),
// the two terms as one packed FP32x2 value.
//
// For c >= 0 both terms are >= 0 and as accurate relative to themselves as
// their coefficients: x + z g >= 2/3 c_1 + (c_0 + c_2) g / 6, and a lone
// coefficient comes out as its weight, s^3 / 6 at the end of its support.  The
// transverse weights are >= 0 too (the FMA that computes their argument clamps
// it to [0, 1]), so A c >= 0.  The powers of t - 1/2, which cost the same,
// cancel at the ends of a support: an absolute error of 6e-9 of the
// coefficient there, and negative projections of non-negative coefficients.
//
// The footprint form (march in spl_march.cuh) carries an (n+1)^3 register
// window that an event shifts by selects and flushes face by face; that is
// half of its instructions, and it must keep the adjoint's order.  Here a
// piece loads its (n+1)^2 columns afresh, always as aligned 16-byte vectors
// (neighbouring lanes and successive pieces share them in L1), so there is
// no window to shift, no face to pick, and a piece does not depend on the
// one before: pieces of one ray may be walked by several threads.
//
// Bound by the FMA pipe (64 % busy) and the latency of a piece's loads at 16
// warps per SM; 8 views of the 512^3 helical workload take 44.5 ms with the
// resampling (the footprint form 73 ms), 120 views of the 256^3 cone 86 ms (149),
// 64 general parallel views of 128^3 5.0 ms (8.9; linear 0.97 and 2.2), quadratic
// 180 x 180 x 50 4.2 ms (5.0).  The relative error against FP64 is 2.7e-8 (1.25e-7
// cubic, 4.3e-8 linear and quadratic).
#include <math.h>

#include <new>

#include "spl_host.h"
#include "spl_line.cuh"

namespace spl {

// The transverse axes of dominant axis d: p (rows) and q (contiguous).  q is
// z where it can be: the detector columns of tilt series and of circular and
// helical orbits about z run along it, and eight lanes along q then load one
// run of columns (see line_lanes_along_v).
__host__ __device__ constexpr int line_p(int d) { return d == 1 ? 0 : 1; }
__host__ __device__ constexpr int line_q(int d) { return d == 2 ? 0 : 2; }

// Resampled array of axis d at degree n: cells c = 0 .. n_d + n - 1, columns
// padded by n zeros on every side (a piece's window then never leaves the
// array).  The row stride is 3 vectors above a multiple of 8: lanes of a
// warp that sit in neighbouring rows or cells then load from different banks
// (8 helical views 51.3 ms with rows on 128-byte boundaries, 49.7 with 3; 64
// general parallel views 5.72 and 4.99 ms).
struct LineDims {
    int nd, np, nq;
};
__host__ __device__ inline LineDims line_dims(const int (&n)[3], int d, int degree)
{
    LineDims L;
    L.nd = sel3(d, n[0], n[1], n[2]) + degree;
    L.np = sel3(line_p(d), n[0], n[1], n[2]) + 2 * degree;
    L.nq = (sel3(line_q(d), n[0], n[1], n[2]) + 2 * degree + 7) / 8 * 8 + 3;
    return L;
}

template <int N> struct LineVec { using T = float4; };
template <> struct LineVec<1> { using T = float2; };

struct LineArrays {
    void *a[3];  // per dominant axis, NULL where no ray has it
};

// ---------------------------------------------------------------- resampling
// x, y, z, w of a cell's coefficients.  Differences first and halves before
// their sum: neighbours of any size do not overflow, and a zero neighbour leaves
// no rounding of the others.  (A division: 1/6 rounded to FP32 would scale
// every value by 1 + 3e-8.)  A coefficient that is not finite would meet its own
// negative in z and w: such a cell is the sum of its coefficients.
template <int N>
__device__ __forceinline__ typename LineVec<N>::T line_cell(const float (&c)[N + 1])
{
    if constexpr (N == 1) {
        return make_float2(c[0], c[1]);
    } else {
        const float l = 0.5f * (c[0] - c[1]), r = 0.5f * (c[2] - c[1]);
        float4 v;
        if constexpr (N == 2)
            v = make_float4(c[1], 0.0f, l, r);
        else
            v = make_float4(c[1], c[2], __fdiv_rn(l + r, 3.0f), __fdiv_rn(0.5f * (c[3] - c[2]) - r, 3.0f));
        if (!isfinite(v.z) || !isfinite(v.w)) {
            const float t = N == 2 ? (c[0] + c[1]) + c[2] : (c[0] + c[1]) + (c[2] + c[N]);
            v = make_float4(t, N == 2 ? 0.0f : t, 0.0f, 0.0f);
        }
        return v;
    }
}

// One thread per column (ip, iq) and chunk of kLineChunk cells, sliding
// along d: one load per cell.  blockIdx.z: (axis, chunk).
constexpr int kLineChunk = 32;
template <int N>
__global__ void __launch_bounds__(256) k_line_resample(DevGeom g, const float *__restrict__ c, LineArrays out, int3 zc)
{
    int d = 0, z = blockIdx.z;
    if (z >= zc.x) {
        z -= zc.x;
        d = 1;
        if (z >= zc.y) {
            z -= zc.y;
            d = 2;
        }
    }
    const LineDims L = line_dims(g.n, d, N);
    const int iq = blockIdx.x * 32 + (threadIdx.x & 31), ip = blockIdx.y * 8 + (threadIdx.x >> 5);
    const int c0 = z * kLineChunk;
    if (iq >= L.nq || ip >= L.np || c0 >= L.nd) return;
    const long long sy = g.n[0], sz = (long long)g.n[0] * g.n[1];
    const int nd = L.nd - N, np = L.np - 2 * N, nq = sel3(line_q(d), g.n[0], g.n[1], g.n[2]);
    auto stride = [&](int e) { return e == 0 ? 1LL : (e == 1 ? sy : sz); };
    const long long sd = stride(d), sp = stride(line_p(d)), sq = stride(line_q(d));
    const bool in = ip >= N && ip - N < np && iq >= N && iq - N < nq;
    const float *src = c + (in ? (ip - N) * sp + (iq - N) * sq : 0);
    typename LineVec<N>::T *o =
        reinterpret_cast<typename LineVec<N>::T *>(d == 0 ? out.a[0] : (d == 1 ? out.a[1] : out.a[2])) +
        ((long long)c0 * L.np + ip) * L.nq + iq;
    const long long so = (long long)L.np * L.nq;
    float w[N + 1];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int l = c0 - N + i;  // cell c0 holds l = c0 - N .. c0
        w[i + 1] = in && l >= 0 && l < nd ? __ldg(src + l * sd) : 0.0f;
    }
    const int c1 = min(c0 + kLineChunk, L.nd);
#pragma unroll 4
    for (int cc = c0; cc < c1; ++cc) {
#pragma unroll
        for (int i = 0; i < N; ++i) w[i] = w[i + 1];
        w[N] = in && cc < nd ? __ldg(src + cc * sd) : 0.0f;
        *o = line_cell<N>(w);
        o += so;
    }
}

// ---------------------------------------------------------------- ray set-up
// A ray, in shared memory: set up by one thread, read by the 2^ls threads
// that share it.
struct __align__(16) LineRay {
    long long A, B;           // v_p, v_q at the start of cell c
    long long RA, RB;         // and their steps
    float ia, ib;             // reciprocals of ra, rb
    float ea, eb;             // the fraction at which the ray leaves its cell: 1 (r > 0), 0 (r < 0)
    float ra, rb;             // steps per cell
    float scale, scale_lo;    // 1 / |w_d| as a sum of two floats
    int d, c, cl;             // dominant axis, first and last cell (none: c > cl)
    int four;                 // cubic: every piece takes four Gauss nodes (line_four)
};

// The line {s + t w} (w of any length).  The two orientations of a line are
// the same line: w_d > 0 is implied by dividing by w_d, and the transverse
// steps keep their signs.  FP64, about 45 operations; GB300 has 1/64 of the
// FP32 rate for them, so a ray is set up once for all its threads.  L comes
// with an empty cell range and keeps it when the line meets no support.
template <int N>
__device__ __forceinline__ void line_setup(const DevGeom &g, const double (&s)[3], const double (&w)[3], LineRay &L)
{
    constexpr double W = 0.5 * (N + 1);
    int d = 0;
    if (fabs(w[1]) > fabs(w[d])) d = 1;
    if (fabs(w[2]) > fabs(w[d])) d = 2;
    L.d = d;
    // p and q by selects (no local-memory indexing)
    const int ap = line_p(d), aq = line_q(d);
    const double u0 = s[0] - g.org[0], u1 = s[1] - g.org[1], u2 = s[2] - g.org[2];
    const double wd = sel3(d, w[0], w[1], w[2]), wp = sel3(ap, w[0], w[1], w[2]), wq = sel3(aq, w[0], w[1], w[2]);
    const double sd = sel3(d, u0, u1, u2), sp = sel3(ap, u0, u1, u2), sq = sel3(aq, u0, u1, u2);
    const int nd = sel3(d, g.n[0], g.n[1], g.n[2]), np = sel3(ap, g.n[0], g.n[1], g.n[2]),
              nq = sel3(aq, g.n[0], g.n[1], g.n[2]);
    const double iw = 1.0 / wd;
    double ra = wp * iw, rb = wq * iw;
    // steps below 1e-30 move nothing over 2048 cells
    if (fabs(ra) < 1e-30) ra = 0.0;
    if (fabs(rb) < 1e-30) rb = 0.0;
    // |w| / |w_d| = sqrt(1 + ra^2 + rb^2): the FP32 root and its correction
    // from the FP64 residual
    const double q2 = fma(ra, ra, fma(rb, rb, 1.0));
    L.scale = sqrtf((float)q2);
    L.scale_lo = fmaf(-weight_excess<N>(2), L.scale, (float)fma(-(double)L.scale, (double)L.scale, q2) * (0.5f / L.scale));
    // transverse coordinates at v_d = 0
    const double a0 = fma(-(W + sd), ra, sp) + W, b0 = fma(-(W + sd), rb, sq) + W;
    L.ra = (float)ra;
    L.rb = (float)rb;
    if (N == 3) L.four = line_four(L.ra, L.rb);
    // an axis that the ray does not move along: crossing at 3 - fraction, never inside a cell
    L.ia = ra != 0.0 ? 1.0f / L.ra : 1.0f;
    L.ib = rb != 0.0 ? 1.0f / L.rb : 1.0f;
    L.ea = ra != 0.0 ? (ra > 0.0 ? 1.0f : 0.0f) : 3.0f;
    L.eb = rb != 0.0 ? (rb > 0.0 ? 1.0f : 0.0f) : 3.0f;
    // cells whose window can hold a basis: v_p in (0, n_p + N), v_q in
    // (0, n_q + N); one cell of margin (the bounds are FP32 quotients)
    float vmin = 0.0f, vmax = (float)(nd + N);
    if (ra != 0.0) {
        const float t0 = (float)(0.0 - a0) * L.ia, t1 = (float)((double)(np + N) - a0) * L.ia;
        vmin = fmaxf(vmin, fminf(t0, t1));
        vmax = fminf(vmax, fmaxf(t0, t1));
    } else if (!(a0 > 0.0 && a0 < (double)(np + N))) {
        return;
    }
    if (rb != 0.0) {
        const float t0 = (float)(0.0 - b0) * L.ib, t1 = (float)((double)(nq + N) - b0) * L.ib;
        vmin = fmaxf(vmin, fminf(t0, t1));
        vmax = fminf(vmax, fmaxf(t0, t1));
    } else if (!(b0 > 0.0 && b0 < (double)(nq + N))) {
        return;
    }
    if (!(vmax >= vmin - 1.0f)) return;
    const int c = max((int)floorf(vmin) - 1, 0);
    L.c = c;
    L.cl = min((int)floorf(vmax) + 1, nd + N - 1);
    constexpr double kOne = (double)(1LL << kLineFrac);
    L.RA = __double2ll_rn(ra * kOne);
    L.RB = __double2ll_rn(rb * kOne);
    L.A = __double2ll_rn(fma((double)c, ra, a0) * kOne);
    L.B = __double2ll_rn(fma((double)c, rb, b0) * kOne);
}

// ---------------------------------------------------------------- the march
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }

// Integral of f over part `seg` of 2^ls equal parts of the cells of L, in
// units of the d axis (times scale outside), as the FP32 sum over the pieces
// and its Kahan compensation (the integral is sum - comp).  Returns false if
// the event bound was reached.
template <int N>
__device__ __forceinline__ bool line_march(const LineRay &L, int seg, int ls, const LineArrays &arr, const int (&n)[3],
                                           const QuadRule &qr, bool kahan, float &sum, float &comp)
{
    using V = typename LineVec<N>::T;
    constexpr int M = GL<N>::M;
    constexpr bool KEEP = N < 3;  // the events' constants in registers
    sum = comp = 0.0f;
    const int cells = L.cl - L.c + 1, k0 = (int)(((long long)cells * seg) >> ls),
              k1 = (int)(((long long)cells * (seg + 1)) >> ls);
    const bool four = N == 3 && __all_sync(0xffffffffu, k0 >= k1 || L.four);
    if (k0 >= k1) return true;
    const int d = L.d;
    long long A = L.A + L.RA * k0, B = L.B + L.RB * k0;
    int left = k1 - k0;  // cells to go
    const float ra = L.ra, rb = L.rb;
    const LineDims D = line_dims(n, d, N);
    const V *__restrict__ P = reinterpret_cast<const V *>(sel3(d, arr.a[0], arr.a[1], arr.a[2]));
    if (!P) return false;  // an axis that line_axes ruled out (not expected)
    const unsigned lim_p = (unsigned)(D.np - N), lim_q = (unsigned)(sel3(line_q(d), n[0], n[1], n[2]) + N);
    const size_t slab = (size_t)D.np * D.nq;
    const V *row = P + (size_t)(L.c + k0) * slab;
    uint4 kr, ke;
    if (KEEP) {
        kr = lds128(&L.RA);
        ke = lds128(&L.ia);
    }
    int QA, QB;
    float ga, gb, ta, tb, t0;
    // position at the cell's start: column (QA, QB) and the fractions; ta, tb:
    // the crossings (beyond 1: none)
    auto cell = [&]() {
        constexpr float kUnit = 1.0f / 4294967296.0f;
        QA = (int)(A >> kLineFrac);
        QB = (int)(B >> kLineFrac);
        ga = __uint2float_rn((unsigned)(A >> (kLineFrac - 32))) * kUnit;
        gb = __uint2float_rn((unsigned)(B >> (kLineFrac - 32))) * kUnit;
        const uint4 e = KEEP ? ke : lds128(&L.ia);
        ta = (__uint_as_float(e.z) - ga) * __uint_as_float(e.x);
        tb = (__uint_as_float(e.w) - gb) * __uint_as_float(e.y);
        t0 = 0.0f;
    };
    cell();
    int ev = 0;
#pragma unroll 1
    while (true) {
        const float t1 = fminf(fminf(ta, tb), 1.0f);
        if (t1 > t0 && (unsigned)QA < lim_p && (unsigned)QB < lim_q) {
            const float half = 0.5f * (t1 - t0), mid = 0.5f * (t0 + t1);
            V col[N + 1][N + 1];
            const V *r = row + ((unsigned)QA * (unsigned)D.nq + (unsigned)QB);
#pragma unroll
            for (int i = 0; i <= N; ++i)
#pragma unroll
                for (int k = 0; k <= N; ++k) col[i][k] = __ldg(r + (size_t)i * D.nq + k);
            float S = 0.0f;
            auto node = [&](float x, float wt) {
                const float t = fmaf(half, x, mid);
                const float2 st = make_float2(1.0f - t, t), gg = N == 3 ? __fmul2_rn(st, st) : st;
                float wa[N + 1], wb[N + 1];
                bweights<N>(__saturatef(fmaf(ra, t, ga)), wa);
                bweights<N>(__saturatef(fmaf(rb, t, gb)), wb);
                float2 h = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int i = 0; i <= N; ++i) {
                    float2 gk;
#pragma unroll
                    for (int k = 0; k <= N; ++k) {
                        float2 e = N == 2 ? dup(col[i][k].x) : make_float2(col[i][k].x, col[i][k].y);
                        if constexpr (N > 1) e = __ffma2_rn(make_float2(col[i][k].z, col[i][k].w), gg, e);
                        gk = k == 0 ? __fmul2_rn(dup(wb[0]), e) : __ffma2_rn(dup(wb[k]), e, gk);
                    }
                    h = i == 0 ? __fmul2_rn(dup(wa[0]), gk) : __ffma2_rn(dup(wa[i]), gk, h);
                }
                // (one sum of whole nodes: a sum for each term rounds more, 2.81e-8 of
                // the cone's forward against 2.68e-8)
                S = fmaf(wt, fmaf(st.x, h.x, st.y * h.y), S);
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
            const float v = half * S;
            if (kahan) kahan_add(sum, comp, v);
            else sum += v;
        }
        t0 = fmaxf(t0, t1);
        if (++ev > qr.cap) return false;
        const bool evA = ta <= tb && ta < 1.0f, evB = !evA && tb < 1.0f;
        if (evA || evB) {
            // the column's neighbour along the crossed axis, once per cell
            const int step = (evA ? ra : rb) > 0.0f ? 1 : -1;
            QA += evA ? step : 0;
            ga -= evA ? (float)step : 0.0f;
            ta = evA ? 2.0f : ta;
            QB += evB ? step : 0;
            gb -= evB ? (float)step : 0.0f;
            tb = evB ? 2.0f : tb;
        } else {
            if (--left == 0) break;
            const uint4 e = KEEP ? kr : lds128(&L.RA);
            A += (long long)(((unsigned long long)e.y << 32) | e.x);
            B += (long long)(((unsigned long long)e.w << 32) | e.z);
            row += slab;
            cell();
            ev = 0;
        }
    }
    return true;
}

// ---------------------------------------------------------------- kernels
// blocks per SM the registers are sized for
template <int N> struct LineBlocks { static constexpr int value = N == 3 ? 4 : (N == 2 ? 5 : 8); };

// The value of thread (seg, ray p of the block): the march over its share of
// the ray's cells, and the sum of the ray's 2^ls shares (adjacent lanes; every
// lane of the warp calls this).  The shares and the scale are carried as
// float pairs and rounded once at the end: rounded one by one they would
// cost as much accuracy as the march itself (5.1e-8 against 2.8e-8).
template <int N>
__device__ __forceinline__ float line_value(const DevGeom &g, const LineRay &L, const LineArrays &arr,
                                            const QuadRule &qr, int kahan, int seg, int ls)
{
    float hi, lo;
    if (!line_march<N>(L, seg, ls, arr, g.n, qr, kahan != 0, hi, lo)) atomicOr(g.err, 1);
    lo = -lo;
    for (int o = 1; o < (1 << ls); o <<= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, o), l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        const float s = __fadd_rn(hi, h2), bb = __fsub_rn(s, hi);  // TwoSum
        lo += l2 + __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(h2, bb));
        hi = s;
    }
    const float p = __fmul_rn(hi, L.scale);
    if (!isfinite(p)) return p;  // (its corrections would be inf - inf)
    return p + fmaf(hi, L.scale_lo, fmaf(lo, L.scale, fmaf(hi, L.scale, -p)));
}

// Whether a warp's eight consecutive lanes run along detector v (4 x 8
// pixels) or u (8 x 4): along the axis that moves more along q, so that they
// load one run of columns (8 cone views 7.9 ms against 6.5 the other way
// round, 8 helical views 99 against 51).  Decided for the view's central ray.
__device__ __forceinline__ bool line_lanes_along_v(const DevGeom &g, const ViewPose &P)
{
    float w[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) w[e] = fabsf((float)(g.kind == SPL_PARALLEL ? P.src[e] : P.dc[e] - P.src[e]));
    const int d = w[1] > w[0] ? (w[2] > w[1] ? 2 : 1) : (w[2] > w[0] ? 2 : 0);
    const int q = line_q(d);
    return fabs(q == 2 ? P.dv[2] : P.dv[0]) >= fabs(q == 2 ? P.du[2] : P.du[0]);
}

// view geometries: view blockIdx.z (of order[], when given)
template <int N>
__global__ void __launch_bounds__(128, LineBlocks<N>::value)
    k_line_views(DevGeom g, LineArrays arr, float *__restrict__ y, QuadRule qr, int kahan, const int *order, int ls)
{
    const int seg = threadIdx.x & ((1 << ls) - 1), p = threadIdx.x >> ls;
    const int k = order ? order[blockIdx.z] : (int)blockIdx.z;
    const bool along_v = line_lanes_along_v(g, g.views[k]);
    __shared__ LineRay rays[128];
    // thread t sets up ray t of the block
    const int t = threadIdx.x;
    if (t < (128 >> ls)) {
        int u, v;
        line_tile(t, ls, along_v, u, v);
        rays[t].c = 0;
        rays[t].cl = -1;
        if (u < g.nu && v < g.nv) {
            double s[3], w[3];
            line_pixel(g, k, u, v, s, w);
            line_setup<N>(g, s, w, rays[t]);
        }
    }
    if (ls == 0) __syncwarp();
    else __syncthreads();
    int iu, iv;
    line_tile(p, ls, along_v, iu, iv);
    const bool in = iu < g.nu && iv < g.nv;
    const float v = line_value<N>(g, rays[p], arr, qr, kahan, seg, ls);
    if (seg == 0 && in) y[((long long)k * g.nv + iv) * g.nu + iu] = v;
}

template <int N>
__global__ void __launch_bounds__(128, LineBlocks<N>::value)
    k_line_rays(DevGeom g, LineArrays arr, float *__restrict__ y, QuadRule qr, int kahan, int ls)
{
    __shared__ LineRay rays[128];
    const long long r0 = ((long long)blockIdx.x * 128) >> ls;
    const int t = threadIdx.x, p = t >> ls, seg = t & ((1 << ls) - 1);
    if (t < (128 >> ls)) {
        rays[t].c = 0;
        rays[t].cl = -1;
        if (r0 + t < g.n_rays) {
            double s[3], w[3];
            explicit_ray(g, r0 + t, s, w);
            line_setup<N>(g, s, w, rays[t]);
        }
    }
    __syncthreads();
    const float v = line_value<N>(g, rays[p], arr, qr, kahan, seg, ls);
    if (seg == 0 && r0 + p < g.n_rays) y[r0 + p] = v;
}

// ---------------------------------------------------------------- host side
// The resampled arrays of a geometry, one block for the largest degree that
// spl_prepare has been asked for; forwards take turns on it (ForwardTurn).
struct LineScratch {
    unsigned mask;   // axes that can be the dominant one of a ray
    size_t need[4];  // bytes of a degree's arrays, 0 where it keeps the footprint form
    void *block;
    size_t bytes;
};

// Where the resampled form is the faster one (both sides measured on GB300):
//  * the arrays are written once per call, 4.7e-12 s a vector, and a piece of
//    a view's ray costs 2.9e-11 s in the footprint form and 1.9e-11 s here:
//    it pays from half a piece per vector on, and a ray crosses about half of
//    nx + ny + nz cells (400^3, rays times nx + ny + nz per vector, footprint form
//    and this one: cubic 0.54 1.21 and 1.41 ms, 0.95 1.77 and 1.70, 1.9 2.82 and
//    2.26; linear 0.97 0.53 and 0.66, 1.9 0.79 and 0.80, 3.8 1.44 and 1.18);
//  * explicit rays that do not lie side by side (spl_geometry::scattered): every
//    lane loads its own 32-byte sectors, and the arrays have to stay mostly in
//    the L2 (135 MB).  300 000 and 600 000 random rays, gain over the footprint
//    form: cubic 176^3 (292 MB) 1.35 1.36, 192^3 (376 MB) 1.23 1.19, 208^3
//    (475 MB) 0.94 0.84; quadratic 144^3 (161 MB) 1.06 1.07, 160^3 (218 MB) 1.00
//    1.00, 176^3 (288 MB) 0.93 0.93; linear 208^3 (231 MB) 1.19 1.04, 224^3
//    (287 MB) 1.11 0.95, 256^3 (425 MB) 0.96 0.81.  Rays side by side gain 1.1 to
//    2.2 up to 384^3 (2.9 GB), like those of views;
//  * all three axes of a cubic 512^3 grid take 6.7 GB; beyond 24 GB, or a quarter
//    of the memory that is free, the scratch is out of proportion.
constexpr size_t kLineMaxBytes = (size_t)24 << 30, kLineSmallBytes = (size_t)1 << 30;
constexpr double kLineScatteredL2[4] = {0.0, 1.75, 1.5, 3.0};  // most bytes in L2s, per degree

// Axes that can be the dominant one of a line of the geometry (a superset).
static unsigned line_axes(const spl_geometry *g, const double *ray_dirs)
{
    unsigned mask = 0;
    line_bounds(g, ray_dirs, [&](const double (&lo)[3], const double (&hi)[3]) {
        for (int e = 0; e < 3; ++e) {
            bool can = true;
            for (int f = 0; f < 3; ++f) can = can && hi[e] * (1.0 + 1e-9) >= lo[f];
            if (can) mask |= 1u << e;
        }
        return mask != 7u;
    });
    return mask;
}

// Byte offsets of the axes' arrays; returns their end.
static size_t line_offsets(const DevGeom &g, unsigned mask, int degree, size_t (&off)[3])
{
    size_t end = 0;
    for (int d = 0; d < 3; ++d) {
        off[d] = end;
        if (!((mask >> d) & 1u)) continue;
        const LineDims L = line_dims(g.n, d, degree);
        const size_t vec = degree == 1 ? sizeof(float2) : sizeof(float4);
        end += ((size_t)L.nd * L.np * L.nq * vec + 255) & ~(size_t)255;
    }
    return end;
}

spl_status line_create(spl_geometry *g, const double *ray_dirs)
{
    const DevGeom &dg = g->dev;
    g->line = nullptr;
    // parallel views of the flat class take the plane matrices or the flat march
    if (dg.n_rays == 0 || (dg.kind == SPL_PARALLEL && dg.n_flat == dg.n_views)) return SPL_OK;
    LineScratch *ls = new (std::nothrow) LineScratch();
    if (!ls) return fail(SPL_ERR_OOM, "host allocation failed");
    ls->mask = line_axes(g, ray_dirs);
    ls->block = nullptr;
    ls->bytes = 0;
    const long long marched = dg.kind == SPL_PARALLEL ? (long long)(dg.n_views - dg.n_flat) * dg.nu * dg.nv : dg.n_rays;
    const double cells = (double)marched * (dg.n[0] + dg.n[1] + dg.n[2]);
    for (int n = 0; n < 4; ++n) {
        size_t off[3];
        const size_t need = n == 0 ? 0 : line_offsets(dg, ls->mask, n, off);
        const double most = g->scattered ? kLineScatteredL2[n] * (double)l2_bytes() : (double)kLineMaxBytes;
        const double vectors = (double)need / (n == 1 ? sizeof(float2) : sizeof(float4));
        ls->need[n] = (double)need <= most && cells >= vectors ? need : 0;
    }
    g->line = ls;
    return SPL_OK;
}

void line_free(LineScratch *ls)
{
    if (!ls) return;
    cudaFree(ls->block);
    delete ls;
}

spl_status line_prepare(spl_geometry *g, int degree, cudaStream_t st)
{
    LineScratch *ls = g->line;
    // (no allocation into a capture: a captured forward has no use for it)
    if (!ls || ls->need[degree] == 0 || stream_captures(st)) return SPL_OK;
    std::lock_guard<std::mutex> lock(g->turn->mu);
    if (ls->bytes >= ls->need[degree]) return SPL_OK;
    // a large scratch that takes more than a quarter of what is free is left out
    // (the query takes 0.2 ms)
    spl_status s = SPL_OK;
    if (ls->need[degree] > kLineSmallBytes) {
        size_t free_bytes = 0, total = 0;
        s = cuda_check(cudaMemGetInfo(&free_bytes, &total), "memory query");
        if (s != SPL_OK) return s;
        if (ls->need[degree] > free_bytes / 4) return SPL_OK;
    }
    // the block of a lower degree may still be in use
    if (ls->block && g->turn->used) s = cuda_check(cudaEventSynchronize(g->turn->last), "line scratch wait");
    if (s != SPL_OK) return s;
    void *block = nullptr;
    if (cudaMalloc(&block, ls->need[degree]) != cudaSuccess) {
        cudaGetLastError();
        return SPL_OK;
    }
    cudaFree(ls->block);
    ls->block = block;
    ls->bytes = ls->need[degree];
    return SPL_OK;
}

bool line_usable(const spl_geometry *g, int degree, bool captured)
{
    // a captured call takes no turn against calls outside the graph: it keeps
    // the footprint form, which has no scratch
    const LineScratch *ls = g->line;
    return ls && !captured && ls->need[degree] > 0 && ls->bytes >= ls->need[degree];
}

template <int N>
static spl_status line_forward_n(const spl_geometry *g, int kahan, const float *c, float *y, cudaStream_t st)
{
    const DevGeom &dg = g->dev;
    const LineScratch &S = *g->line;
    const QuadRule qr = quad_rule(N);
    LineArrays arr;
    size_t off[3];
    line_offsets(dg, S.mask, N, off);
    for (int d = 0; d < 3; ++d) arr.a[d] = ((S.mask >> d) & 1u) ? (char *)S.block + off[d] : nullptr;
    int gx = 0, gy = 0, zc[3];
    for (int d = 0; d < 3; ++d) {
        zc[d] = 0;
        if (!arr.a[d]) continue;
        const LineDims L = line_dims(dg.n, d, N);
        zc[d] = (L.nd + kLineChunk - 1) / kLineChunk;
        gx = (L.nq + 31) / 32 > gx ? (L.nq + 31) / 32 : gx;
        gy = (L.np + 7) / 8 > gy ? (L.np + 7) / 8 : gy;
    }
    k_line_resample<N><<<dim3(gx, gy, zc[0] + zc[1] + zc[2]), 256, 0, st>>>(dg, c, arr, make_int3(zc[0], zc[1], zc[2]));
    if (dg.kind == SPL_RAYS) {
        const int ls = line_split(dg.n_rays, LineBlocks<N>::value);
        const long long blocks = ((dg.n_rays << ls) + 127) / 128;
        k_line_rays<N><<<(unsigned)blocks, 128, 0, st>>>(dg, arr, y, qr, kahan, ls);
    } else {
        const int v0 = dg.kind == SPL_PARALLEL ? dg.n_flat : 0, nview = dg.n_views - v0;
        const int *order = dg.kind == SPL_PARALLEL ? dg.view_order + v0 : nullptr;
        const int ls = line_split((long long)nview * dg.nu * dg.nv, LineBlocks<N>::value);
        k_line_views<N><<<line_grid(dg, nview, ls), 128, 0, st>>>(dg, arr, y, qr, kahan, order, ls);
    }
    return cuda_check(cudaGetLastError(), "line forward launch");
}

spl_status line_forward(const spl_geometry *g, int degree, int kahan, const float *c, float *y, cudaStream_t st)
{
    switch (degree) {
    case 1: return line_forward_n<1>(g, kahan, c, y, st);
    case 2: return line_forward_n<2>(g, kahan, c, y, st);
    default: return line_forward_n<3>(g, kahan, c, y, st);
    }
}

}  // namespace spl
