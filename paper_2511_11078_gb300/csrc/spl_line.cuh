// spl_line.cuh -- shared by the forward on resampled coefficients (line.cu)
// and the scatter adjoint (scatter.cu): fixed-point ray positions, the rule
// for four Gauss nodes, the block's pixels and the number of threads per ray.
#pragma once

#include "spl_host.h"

namespace spl {

// (selects: a run-time index would put the array into local memory)
template <class T> __host__ __device__ inline T sel3(int i, const T &a, const T &b, const T &c)
{
    return i == 0 ? a : (i == 1 ? b : c);
}

// Transverse coordinates are carried as 64-bit fixed point with kLineFrac
// fraction bits (and 15 bits and a sign for cells: the grid has at most 2048,
// and a ray is marched where it meets it).  The start is the FP64 value, exact
// to 2^-43, and the step is off by at most 2^-49 per cell, 2^-38 over the
// longest ray; a cell takes its fraction's upper 32 bits.  One 64-bit add per
// cell.
constexpr int kLineFrac = 48;

// The FP32 constants 2/3 and 1/6 of the cubic weights (bweights<3>) are
// 1.987e-8 and 4.97e-9 too large, so the four weights of an axis sum to
// 1 + 2 (1.987e-8) + 4.97e-9 (g^3 + t^3), on average 1 + 4.22e-8, and an
// integral over `axes` such axes comes out that much too large.  The ray's
// scale takes it out (it was most of the forward's error against FP64).
template <int N> __device__ __forceinline__ constexpr float weight_excess(int axes) { return N == 3 ? 4.22e-8f * axes : 0.0f; }

// Whether every piece of a cubic ray takes the 4-node Gauss rule.  It is exact
// to degree 7; of the degree-9 product of a piece of length h <= 1 it misses
// only the coefficient C8 of the 8th power about the piece's middle (the 9th is
// odd there), by
//   e8 (h/2)^9 C8,  e8 = 2^9 (4!)^4 / (9 (8!)^2) = 0.01161,
// and C8 = D2 A3 B3 + D3 A2 B3 + D3 A3 B2 with |D3| <= 1/2, |A3| <= ra^3 / 2,
// |B3| <= rb^3 / 2 the third- and |D2| <= 1, |A2| <= ra^2, |B2| <= rb^2 the
// second-order coefficients of the three weights, so a piece misses at most
// 5.67e-6 h^9 (ra rb + ra + rb) ra^2 rb^2 of a footprint.  The rule is taken
// where that is below 2^-28 at h = 1, an eighth of an ulp of the footprint's
// peak (0.44) for each of its pieces (up to a dozen, most of them far shorter):
// the difference drowns in the FP32 rounding of the sums (A^T of a 128^3 cone
// against FP64: 1.359e-7 with the rule, 1.373e-7 with five nodes for all).  It
// is an absolute bound: where a ray clips the corner of a support, a footprint
// of 1e-8 of the peak can miss 1e-4 of itself.
// A warp takes it when all its rays do, decided once where the warp is whole,
// so a ray's value depends on the rays that share its warp and on nothing else;
// half of the warps of a cone or helical orbit do.  Five nodes for all: 8
// helical views A 44.4 -> 50.9 ms, A^T 54.9 -> 60.3, 8 cone views 6.16 -> 6.45 and
// 7.35 -> 7.68.  A rule for each piece and lane (selected nodes, the fifth in a
// branch): 44.5, 55.9, 6.15, 7.50.
__device__ __forceinline__ bool line_four(float ra, float rb)
{
    ra = fabsf(ra);
    rb = fabsf(rb);
    return 5.67e-6f * 0x1p28f * (fmaf(ra, rb, ra) + rb) * (ra * ra) * (rb * rb) <= 1.0f;
}

// 16 bytes of a ray, not to be kept in registers: next to 64 column values
// the cubic march has none for the constants that only its events need (with
// them in registers it spills: 8 helical views 51.9 ms, 49.5 without), so
// the load is volatile and stays in the loop.
__device__ __forceinline__ uint4 lds128(const void *p)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
    return v;
}

// Pixel p of a block's tile: 16 x 8 pixels with one thread a ray, 8 x 8, 8 x 4,
// 4 x 4 with 2, 4, 8 threads a ray.  One thread a ray: a warp covers 4 x 8
// pixels with eight consecutive lanes along v, or 8 x 4 with them along u.
__device__ __forceinline__ void line_tile(int p, int ls, bool along_v, int &iu, int &iv)
{
    const int lane = p & 31, wid = p >> 5;
    if (ls == 0 && along_v) {
        iu = blockIdx.x * 16 + wid * 4 + (lane >> 3);
        iv = blockIdx.y * 8 + (lane & 7);
    } else if (ls == 0) {
        iu = blockIdx.x * 16 + (wid & 1) * 8 + (lane & 7);
        iv = blockIdx.y * 8 + (wid >> 1) * 4 + (lane >> 3);
    } else {
        const int lw = ls == 3 ? 2 : 3;
        iu = (blockIdx.x << lw) + (p & ((1 << lw) - 1));
        iv = blockIdx.y * (ls == 1 ? 8 : 4) + (p >> lw);
    }
}
inline dim3 line_grid(const DevGeom &dg, int views, int ls)
{
    const int tw = ls == 0 ? 16 : (ls == 3 ? 4 : 8), th = ls < 2 ? 8 : 4;
    return dim3((dg.nu + tw - 1) / tw, (dg.nv + th - 1) / th, views);
}

// The line of pixel (u, v) of view k: a point and a direction of any length.
__device__ __forceinline__ void line_pixel(const DevGeom &g, int k, int u, int v, double (&s)[3], double (&w)[3])
{
    const ViewPose &P = g.views[k];
    const double a = u - 0.5 * (g.nu - 1), b = v - 0.5 * (g.nv - 1);
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const double q = fma(b, P.dv[e], fma(a, P.du[e], P.dc[e])), src = P.src[e];
        s[e] = q;
        w[e] = g.kind == SPL_PARALLEL ? src : q - src;
    }
}

// Threads per ray, 2^ls: the fewest that give every SM its resident threads,
// at most 8 (a thread keeps at least a few cells of the ray).
inline int line_split(long long rays, int blocks_per_sm)
{
    const long long fill = (long long)sm_count() * blocks_per_sm * 128;
    int ls = 0;
    while (ls < 3 && (rays << ls) < fill) ++ls;
    return ls;
}

// Bounds lo <= |w_e| <= hi of the direction components over each explicit ray
// or over each view's pixels (taken at its corners: a pixel's direction is
// affine in (u, v)), handed to f until it returns false.
template <class F> inline void line_bounds(const spl_geometry *g, const double *ray_dirs, F f)
{
    const DevGeom &dg = g->dev;
    if (dg.kind == SPL_RAYS) {
        for (long long r = 0; r < dg.n_rays; ++r) {
            double m[3];
            for (int e = 0; e < 3; ++e) m[e] = fabs(ray_dirs[3 * r + e]);
            if (!f(m, m)) return;
        }
        return;
    }
    for (int k = 0; k < dg.n_views; ++k) {
        const ViewPose &P = g->views_host[k];
        double lo[3], hi[3];
        for (int e = 0; e < 3; ++e) {
            double mn = INFINITY, mx = -INFINITY;
            for (int corner = 0; corner < 4; ++corner) {
                const double a = ((corner & 1) ? 0.5 : -0.5) * (dg.nu - 1), b = ((corner & 2) ? 0.5 : -0.5) * (dg.nv - 1);
                const double v = dg.kind == SPL_PARALLEL ? P.src[e] : P.dc[e] + a * P.du[e] + b * P.dv[e] - P.src[e];
                mn = fmin(mn, v);
                mx = fmax(mx, v);
            }
            lo[e] = mn <= 0.0 && mx >= 0.0 ? 0.0 : fmin(fabs(mn), fabs(mx)) * (1.0 - 1e-9);
            hi[e] = fmax(fabs(mn), fabs(mx));
        }
        if (!f(lo, hi)) return;
    }
}

}  // namespace spl
