// mlp.cu -- the learned footprint f_theta (Sec. 2.2) and its training
// (Algorithm 1): parameters, BF16 evaluation copy, batched evaluation on the
// tensor cores, the MLP footprint of spl_footprint, gradients of the L2
// loss and Adam.
//
// Training step (all kernels here, one stream, no host sync):
//   k_train_forward  -- the inference tile (tcgen05 BF16 MMAs) on the batch,
//                       saving pre-activations and the activations that
//                       entered each layer;
//   k_train_backward -- per batch chunk, dL/dz of every layer (FP32, the BF16
//                       roundings passed straight through) and from it
//                       dL/dW = sum_b dz_b x h_b^T and dL/db, into fixed
//                       partial slots;
//   k_train_reduce   -- adds the chunk partials in a fixed order (deterministic)
//                       and the loss;
//   k_adam           -- Adam on the FP32 master copy, then k_prep refreshes
//                       the BF16 evaluation copy.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include "spl_mlp.cuh"
#include "spl_tc.cuh"

namespace spl {

constexpr int kChunkRows = 64;     // rows per weight-gradient partial

}  // namespace spl

struct spl_mlp {
    int degree;
    int max_batch;
    int device;
    int step;
    unsigned long long seed;  // seed of the initial parameters
    float *master;    // [kParams] FP32 master parameters
    float *adam_m;    // [kParams]
    float *adam_v;    // [kParams]
    float *grad;      // [kParams]
    uint32_t *w23;    // evaluation copy, BF16 hidden layers
    float *f32;       // evaluation copy, FP32 first/last layers and biases
    void *tc_img;     // evaluation copy in the tcgen05 tile's operand layout
    float *act;       // [6][max_batch][64] z1 h1 z2 h2 z3 h3
    float *out;       // [max_batch] outputs
    float *part;      // [chunks][kPartStride] weight-gradient partials
    double *loss_part;  // [chunks] loss partials
    int *err;         // device error flag (kErrTimeout: a tensor-core wait gave up)
    void *block;      // single device allocation holding all of the above
};

namespace spl {

MlpDev mlp_dev(const spl_mlp *m)
{
    MlpDev d;
    d.w23 = m->w23;
    d.f32 = m->f32;
    d.tc_img = m->tc_img;
    d.err = m->err;
    return d;
}

// ---------------------------------------------------------------- evaluation copy
__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

__global__ void k_prep(const float *__restrict__ P, uint32_t *__restrict__ w23, float *__restrict__ f32,
                       TcMlpImage *img)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    // the tcgen05 tile's image of the same roundings
    tc_mlp_image(P, *img, i, gridDim.x * blockDim.x);
    // hidden layers: rows of W2 / W3 as BF16 pairs, padded stride
    if (i < 2 * kHid * kRowWords) {
        const int layer = i / (kHid * kRowWords), rem = i % (kHid * kRowWords);
        const int row = rem / kRowWords, w = rem % kRowWords;
        const float *W = P + (layer == 0 ? kOffW2 : kOffW3);
        uint32_t v = 0;
        if (w < kHid / 2) v = pack_bf16(W[row * kHid + 2 * w], W[row * kHid + 2 * w + 1]);
        w23[i] = v;
    }
    if (i < kF32Size) {
        float v;
        if (i < kF32B1) v = bf16r(P[kOffW1 + i]);
        else if (i < kF32B2) v = P[kOffB1 + (i - kF32B1)];
        else if (i < kF32B3) v = P[kOffB2 + (i - kF32B2)];
        else if (i < kF32W4) v = P[kOffB3 + (i - kF32B3)];
        else if (i < kF32B4) v = bf16r(P[kOffW4 + (i - kF32W4)]);
        else v = P[kOffB4];
        f32[i] = v;
    }
}

static spl_status prep(spl_mlp *m, cudaStream_t st)
{
    const int n = 2 * kHid * kRowWords;
    k_prep<<<(n + 255) / 256, 256, 0, st>>>(m->master, m->w23, m->f32, reinterpret_cast<TcMlpImage *>(m->tc_img));
    return cuda_check(cudaGetLastError(), "mlp prep launch");
}

// ---------------------------------------------------------------- batched evaluation
// FROM_WP: rows given as (omega, p) -> canonical features and the exact
// support mask of the basis at the origin; otherwise rows are features.
template <bool FROM_WP>
__global__ void __launch_bounds__(2 * kTcRows, 2) k_mlp_rows(MlpDev w, int degree, long long count,
                                                      const float *__restrict__ a, const float *__restrict__ b,
                                                      float *__restrict__ out)
{
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    TcMlpSmem<1> &S = *reinterpret_cast<TcMlpSmem<1> *>(tc_smem);
    TcTile &T = S.tile[0];
    const int tid = threadIdx.x;
    __shared__ float part[2 * kTcRows];
    tc_mlp_setup(w, S);
    unsigned phase = 0;
    const long long tiles = (count + kTcRows - 1) / kTcRows;
    for (long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const long long r = tile * kTcRows + (tid & (kTcRows - 1));
        float x[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        float mask = 0.0f;
        if (r < count) {
            mask = 1.0f;
            if (FROM_WP) {
                float wv[3], pv[3];
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    wv[e] = a[3 * r + e];
                    pv[e] = b[3 * r + e];
                }
                const float inrm = rsqrtf(wv[0] * wv[0] + wv[1] * wv[1] + wv[2] * wv[2]);
#pragma unroll
                for (int e = 0; e < 3; ++e) wv[e] *= inrm;
                canonical_features_f32(degree, wv, pv, x);
                // exact support: the line p + t w meets the open cube
                // [-W, W]^3 in a segment of positive length
                const float W = 0.5f * (degree + 1);
                float lo = -INFINITY, hi = INFINITY;
                bool in = true;
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    if (wv[e] == 0.0f) {
                        in = in && (pv[e] >= -W && pv[e] < W) && (degree == 0 || pv[e] > -W);
                    } else {
                        const float iw = 1.0f / wv[e];
                        const float t1 = (-W - pv[e]) * iw, t2 = (W - pv[e]) * iw;
                        lo = fmaxf(lo, fminf(t1, t2));
                        hi = fminf(hi, fmaxf(t1, t2));
                    }
                }
                mask = (in && hi > lo) ? 1.0f : 0.0f;
            } else {
#pragma unroll
                for (int e = 0; e < 5; ++e) x[e] = a[5 * r + e];
            }
        }
        float o;
        const bool ok = tc_mlp_tile<2>(S.img, T, tid, 0, true, x, o, phase, part);
        // a tensor-core wait that gave up (not expected) leaves NaN in the
        // rows of the tile, sets the network's error flag and stops the CTA
        const bool bad = __syncthreads_or(!ok);
        if (r < count && tid < kTcRows) out[r] = bad ? __int_as_float(0x7FC00000) : o * mask;
        if (bad) {
            if (threadIdx.x == 0) atomicOr(w.err, kErrTimeout);
            tc_mlp_teardown(S, T, phase, true);
            return;
        }
    }
    tc_mlp_teardown(S, T);
}

static unsigned eval_blocks(long long count)
{
    const long long tiles = (count + kTcRows - 1) / kTcRows;
    const long long cap = 4LL * sm_count();
    return (unsigned)(tiles < cap ? (tiles > 0 ? tiles : 1) : cap);
}

// dynamic shared memory of the tcgen05 row kernels (set once per process)
template <bool FROM_WP> static spl_status rows_smem_attr()
{
    return smem_attr_once((const void *)k_mlp_rows<FROM_WP>, (int)sizeof(TcMlpSmem<1>), "mlp rows smem attribute");
}

spl_status footprint_mlp(const spl_basis_desc *b, long long count, const float *w, const float *p, float *out,
                         cudaStream_t st)
{
    spl_status s = rows_smem_attr<true>();
    if (s != SPL_OK) return s;
    k_mlp_rows<true><<<eval_blocks(count), 2 * kTcRows, sizeof(TcMlpSmem<1>), st>>>(mlp_dev(b->mlp), b->degree, count, w, p,
                                                                             out);
    return cuda_check(cudaGetLastError(), "mlp footprint launch");
}

// ---------------------------------------------------------------- training
__global__ void __launch_bounds__(2 * kTcRows, 2) k_train_forward(MlpDev w, int B, const float *__restrict__ X,
                                                               float *act, float *out, int max_batch)
{
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    TcMlpSmem<1> &S = *reinterpret_cast<TcMlpSmem<1> *>(tc_smem);
    TcTile &T = S.tile[0];
    const int tid = threadIdx.x;
    __shared__ float part[2 * kTcRows];
    tc_mlp_setup(w, S);
    unsigned phase = 0;
    const size_t L = (size_t)max_batch * 64;
    const int tiles = (B + kTcRows - 1) / kTcRows;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int r = tile * kTcRows + (tid & (kTcRows - 1));
        float x[5];
#pragma unroll
        for (int e = 0; e < 5; ++e) x[e] = r < B ? X[5 * r + e] : 0.0f;
        const TcSave sv{act, act + L, act + 2 * L, act + 3 * L, act + 4 * L, act + 5 * L, r < B ? r : -1};
        float o;
        const bool ok = tc_mlp_tile<2, true>(S.img, T, tid, 0, true, x, o, phase, part, &sv);
        // a tensor-core wait that gave up (not expected) leaves NaN outputs,
        // so the loss and the gradient come out NaN, and sets the network's
        // error flag
        const bool bad = __syncthreads_or(!ok);
        if (r < B && tid < kTcRows) out[r] = bad ? __int_as_float(0x7FC00000) : o;
        if (bad) {
            if (threadIdx.x == 0) atomicOr(w.err, kErrTimeout);
            tc_mlp_teardown(S, T, phase, true);
            return;
        }
    }
    tc_mlp_teardown(S, T);
}

__device__ __forceinline__ float silu_grad(float z)
{
    const float s = 1.0f / (1.0f + expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

// Gradients of one batch chunk (64 rows) for L = (1/B) sum (f(x_b) - y_b)^2:
// dL/dz of the three hidden layers, and from each the layer's weight and bias
// gradients, without leaving the block.  A layer is two 64 x 64 x 64 FP32
// products on the chunk's dz: dW[o][i] = sum_r dz[r][o] h[r][i] and the layer
// below's dh[r][i] = sum_o dz[r][o] W[o][i]; dz sits in shared memory in both
// orders, so that every operand of a thread's 4 x 4 outputs is one 16-byte
// load per step.  Weights as used in the forward (BF16-rounded) come from the
// FP32 master rounded on the fly; roundings of activations pass straight
// through.  Rows are summed in order (deterministic).
//
// 8192 rows are 128 blocks, less than one wave: the time is one block's
// latency.  A gradient of 8192 samples went from 82 to 40 us with this kernel
// in place of one thread group per row for dz and 512 blocks for the products,
// which passed dz through memory; 512 threads with 4 x 2 outputs took 41.
constexpr int kBwdThreads = 256;
constexpr int kPartStride = (kParams + 1 + 3) & ~3;  // floats per chunk of partials, 16-byte rows
constexpr int kDzPad = 4;                            // row padding (floats) of the dz arrays
struct __align__(16) BwdSmem {
    float W2[kHid * kHid], W3[kHid * kHid];
    float D[kChunkRows][kHid + kDzPad];   // dz[r][o]
    float DT[kHid][kChunkRows + kDzPad];  // dz[o][r]
    float H[kChunkRows][kHid];            // activations that entered the layer
    float W4[kHid], d4[kChunkRows], X[kChunkRows * kIn];
    double red[kBwdThreads / 32];
};

// sum_k a[k][i0 + i] b[k][j0 + j] for i, j = 0..3 over 64 k; rows of sa, sb floats
__device__ __forceinline__ void product4x4(const float *a, int sa, const float *b, int sb, float (&c)[4][4])
{
    float2 acc[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = make_float2(0.0f, 0.0f);
#pragma unroll 8
    for (int k = 0; k < 64; ++k) {
        const float4 x = *reinterpret_cast<const float4 *>(a + k * sa), y = *reinterpret_cast<const float4 *>(b + k * sb);
        const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            acc[i][0] = __ffma2_rn(make_float2(xs[i], xs[i]), make_float2(y.x, y.y), acc[i][0]);
            acc[i][1] = __ffma2_rn(make_float2(xs[i], xs[i]), make_float2(y.z, y.w), acc[i][1]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        c[i][0] = acc[i][0].x;
        c[i][1] = acc[i][0].y;
        c[i][2] = acc[i][1].x;
        c[i][3] = acc[i][1].y;
    }
}

__global__ void __launch_bounds__(kBwdThreads, 2) k_train_backward(const float *__restrict__ P, int B,
                                                                   const float *__restrict__ X, const float *__restrict__ Y,
                                                                   const float *__restrict__ act,
                                                                   const float *__restrict__ out, float *__restrict__ part,
                                                                   double *__restrict__ loss_part, int max_batch)
{
    extern __shared__ __align__(16) unsigned char bwd_smem[];
    BwdSmem &S = *reinterpret_cast<BwdSmem *>(bwd_smem);
    const int t = threadIdx.x, r0 = blockIdx.x * kChunkRows, nr = min(kChunkRows, B - r0);
    const size_t L = (size_t)max_batch * 64;
    float *dst = part + (size_t)blockIdx.x * kPartStride;
    const int p4 = 4 * (t >> 4), q4 = 4 * (t & 15);  // this thread's 4 x 4 outputs
    // rows p4 .. p4 + 3, columns q4 .. q4 + 3 of an activation array (0 beyond the batch)
    auto rows = [&](const float *src, float4 (&v)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            v[i] = p4 + i < nr ? __ldg(reinterpret_cast<const float4 *>(src + (size_t)(r0 + p4 + i) * 64 + q4))
                               : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    };
    // everything the block reads is requested first
    float4 z3[4], h2[4], z2[4], h1[4], z1[4], h3[4];
    rows(act + 4 * L, z3);
    rows(act + 5 * L, h3);
    rows(act + 3 * L, h2);
    rows(act + 2 * L, z2);
    rows(act + L, h1);
    rows(act, z1);
    for (int i = t; i < kHid * kHid / 4; i += kBwdThreads) {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(P + kOffW2) + i),
                     b = __ldg(reinterpret_cast<const float4 *>(P + kOffW3) + i);
        reinterpret_cast<float4 *>(S.W2)[i] = make_float4(bf16r(a.x), bf16r(a.y), bf16r(a.z), bf16r(a.w));
        reinterpret_cast<float4 *>(S.W3)[i] = make_float4(bf16r(b.x), bf16r(b.y), bf16r(b.z), bf16r(b.w));
    }
    if (t < kHid) S.W4[t] = bf16r(P[kOffW4 + t]);
    for (int i = t; i < kChunkRows * kIn; i += kBwdThreads) S.X[i] = i < nr * kIn ? X[(size_t)r0 * kIn + i] : 0.0f;
    double l2 = 0.0;
    if (t < kChunkRows) {
        const float res = t < nr ? out[r0 + t] - Y[r0 + t] : 0.0f;
        l2 = (double)res * res;
        S.d4[t] = 2.0f * res / (float)B;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l2 += __shfl_down_sync(0xffffffffu, l2, o);
    if ((t & 31) == 0) S.red[t >> 5] = l2;
    auto put = [&](float (&dst_)[kChunkRows][kHid], const float4 (&v)[4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<float4 *>(&dst_[p4 + i][q4]) = v[i];
    };
    // dz of a layer in both orders, and the activations that entered it
    auto put_dz = [&](const float (&d)[4][4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            *reinterpret_cast<float4 *>(&S.D[p4 + i][q4]) = make_float4(d[i][0], d[i][1], d[i][2], d[i][3]);
            *reinterpret_cast<float4 *>(&S.DT[q4 + i][p4]) = make_float4(d[0][i], d[1][i], d[2][i], d[3][i]);
        }
    };
    auto grad_of = [&](const float (&g)[4][4], const float4 (&z)[4], float (&d)[4][4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            d[i][0] = g[i][0] * silu_grad(z[i].x);
            d[i][1] = g[i][1] * silu_grad(z[i].y);
            d[i][2] = g[i][2] * silu_grad(z[i].z);
            d[i][3] = g[i][3] * silu_grad(z[i].w);
        }
    };
    float g[4][4], d[4][4];
    // output layer: dW4 = sum_r d4 h3, db4 = sum_r d4
    put(S.H, h3);
    __syncthreads();
    if (t < kHid) {
        float a = 0.0f;
        for (int r = 0; r < nr; ++r) a = fmaf(S.d4[r], S.H[r][t], a);
        dst[kOffW4 + t] = a;
    } else if (t == kHid) {
        float a = 0.0f;
        for (int r = 0; r < nr; ++r) a += S.d4[r];
        dst[kOffB4] = a;
    } else if (t == kHid + 1) {
        double s = 0.0;
        for (int w = 0; w < kBwdThreads / 32; ++w) s += S.red[w];
        loss_part[blockIdx.x] = s;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) g[i][j] = S.W4[q4 + j] * S.d4[p4 + i];
    grad_of(g, z3, d);
    __syncthreads();
    // a hidden layer: weight gradient, bias gradient, dz of the layer below
    auto layer = [&](const float4 (&h)[4], int offW, int offB, const float *W, const float4 (&zb)[4]) {
        put_dz(d);
        put(S.H, h);
        __syncthreads();
        float w[4][4];
        product4x4(&S.D[0][p4], kHid + kDzPad, &S.H[0][q4], kHid, w);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            *reinterpret_cast<float4 *>(dst + offW + (p4 + i) * kHid + q4) = make_float4(w[i][0], w[i][1], w[i][2], w[i][3]);
        if (t < kHid) {
            float a = 0.0f;
            for (int r = 0; r < kChunkRows; ++r) a += S.D[r][t];
            dst[offB + t] = a;
        }
        product4x4(&S.DT[0][p4], kChunkRows + kDzPad, W + q4, kHid, g);
        grad_of(g, zb, d);
        __syncthreads();
    };
    layer(h2, kOffW3, kOffB3, S.W3, z2);
    layer(h1, kOffW2, kOffB2, S.W2, z1);
    put_dz(d);
    __syncthreads();
    // first layer: inputs e = t / 64 and (t / 64 == 0) 4, the bias with e = 1
    {
        const int o = t & 63, e = t >> 6;
        float a = 0.0f, c = 0.0f;
        for (int r = 0; r < nr; ++r) {
            const float v = S.D[r][o];
            a = fmaf(v, S.X[r * kIn + e], a);
            c = e == 0 ? fmaf(v, S.X[r * kIn + 4], c) : c + v;
        }
        dst[kOffW1 + o * kIn + e] = a;
        if (e == 0) dst[kOffW1 + o * kIn + 4] = c;
        if (e == 1) dst[kOffB1 + o] = c;
    }
}

// Gradient and loss from the partials in a fixed order: block b owns 32
// parameters; warp w sums chunks w, w + 8, ... in order, then warp 0 adds
// the 8 sums in order.  Block 0 also sums the loss partials (thread t:
// partials t, t + 256, ...; then 8 per lane and a fixed shuffle tree).
constexpr int kRedThreads = 256;
__global__ void __launch_bounds__(kRedThreads) k_train_reduce(const float *__restrict__ part, int chunks,
                                                              const double *__restrict__ loss_part, int nloss, int B,
                                                              float *grad, float *loss_out)
{
    __shared__ float ps[kRedThreads / 32][32];
    __shared__ double ls[kRedThreads];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    float acc = 0.0f;
    if (i < kParams)
#pragma unroll 8
        for (int c = w; c < chunks; c += kRedThreads / 32) acc += __ldg(part + (size_t)c * kPartStride + i);
    ps[w][lane] = acc;
    const bool do_loss = blockIdx.x == 0 && loss_out != nullptr;
    if (do_loss) {
        double l = 0.0;
        for (int k = threadIdx.x; k < nloss; k += kRedThreads) l += loss_part[k];
        ls[threadIdx.x] = l;
    }
    __syncthreads();
    if (w == 0) {
        if (i < kParams) {
            float t = 0.0f;
#pragma unroll
            for (int g = 0; g < kRedThreads / 32; ++g) t += ps[g][lane];
            grad[i] = t;
        }
        if (do_loss) {
            double t = 0.0;
#pragma unroll
            for (int k = 0; k < kRedThreads / 32; ++k) t += ls[lane * (kRedThreads / 32) + k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            if (lane == 0) loss_out[0] = (float)(t / (double)B);
        }
    }
}

__global__ void k_adam(float *P, float *m, float *v, const float *__restrict__ g, float lr, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kParams) return;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

static spl_status grad_impl(spl_mlp *m, int B, const float *X, const float *Y, float *grad, float *loss,
                            cudaStream_t st)
{
    const MlpDev w = mlp_dev(m);
    {
        spl_status s = smem_attr_once((const void *)k_train_forward, (int)sizeof(TcMlpSmem<1>),
                                      "train forward smem attribute");
        if (s != SPL_OK) return s;
    }
    k_train_forward<<<eval_blocks(B), 2 * kTcRows, sizeof(TcMlpSmem<1>), st>>>(w, B, X, m->act, m->out, m->max_batch);
    const spl_status sb = smem_attr_once((const void *)k_train_backward, (int)sizeof(BwdSmem), "train backward smem attribute");
    if (sb != SPL_OK) return sb;
    const int chunks = (B + kChunkRows - 1) / kChunkRows;
    k_train_backward<<<chunks, kBwdThreads, sizeof(BwdSmem), st>>>(m->master, B, X, Y, m->act, m->out, m->part, m->loss_part,
                                                                   m->max_batch);
    k_train_reduce<<<(kParams + 31) / 32, kRedThreads, 0, st>>>(m->part, chunks, m->loss_part, chunks, B, grad, loss);
    return cuda_check(cudaGetLastError(), "mlp gradient launch");
}

// SplitMix64 (Steele, Lea and Flood 2014): seeded initial parameters.
static uint64_t splitmix64(uint64_t &x)
{
    uint64_t z = (x += 0x9e3779b97f4a7c15ULL);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

}  // namespace spl

using namespace spl;

extern "C" int spl_mlp_degree(const spl_mlp *m) { return m ? m->degree : -1; }

extern "C" spl_status spl_mlp_create(int degree, int max_batch, unsigned long long seed, spl_mlp **out)
{
    clear_error();
    if (!out) return fail(SPL_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (degree < 0 || degree > 3) return fail(SPL_ERR_ARG, "degree %d not in 0..3", degree);
    if (max_batch < 16 || max_batch > (1 << 22)) return fail(SPL_ERR_ARG, "max_batch %d not in 16..2^22", max_batch);
    spl_mlp *m = (spl_mlp *)calloc(1, sizeof(spl_mlp));
    if (!m) return fail(SPL_ERR_OOM, "host allocation failed");
    m->degree = degree;
    m->max_batch = max_batch;
    m->seed = seed;
    cudaGetDevice(&m->device);
    const int chunks = (max_batch + kChunkRows - 1) / kChunkRows;
    const int nloss = chunks;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += (bytes + 255) & ~(size_t)255;
        return o;
    };
    const size_t o_master = take(kParams * 4), o_m = take(kParams * 4), o_v = take(kParams * 4),
                 o_grad = take(kParams * 4), o_w23 = take(2 * kHid * kRowWords * 4), o_f32 = take(kF32Size * 4),
                 o_img = take(sizeof(TcMlpImage)),
                 o_act = take((size_t)6 * max_batch * 64 * 4), o_out = take((size_t)max_batch * 4),
                 o_part = take((size_t)chunks * kPartStride * 4), o_loss = take((size_t)nloss * 8),
                 o_err = take(sizeof(int));
    void *blk = nullptr;
    cudaError_t ce = cudaMalloc(&blk, off);
    if (ce != cudaSuccess) {
        free(m);
        cudaGetLastError();
        return fail(SPL_ERR_OOM, "cudaMalloc(%zu) failed: %s", off, cudaGetErrorString(ce));
    }
    char *base = (char *)blk;
    m->block = blk;
    m->master = (float *)(base + o_master);
    m->adam_m = (float *)(base + o_m);
    m->adam_v = (float *)(base + o_v);
    m->grad = (float *)(base + o_grad);
    m->w23 = (uint32_t *)(base + o_w23);
    m->f32 = (float *)(base + o_f32);
    m->tc_img = base + o_img;
    m->act = (float *)(base + o_act);
    m->out = (float *)(base + o_out);
    m->part = (float *)(base + o_part);
    m->loss_part = (double *)(base + o_loss);
    m->err = (int *)(base + o_err);
    if (cudaMemset(m->err, 0, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(blk);
        free(m);
        return fail(SPL_ERR_CUDA, "error flag clear failed");
    }
    // seeded uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) for weights and biases
    float *h = (float *)malloc(kParams * sizeof(float));
    if (!h) { cudaFree(blk); free(m); return fail(SPL_ERR_OOM, "host allocation failed"); }
    uint64_t st = seed;
    const int fan_in[4] = {kIn, kHid, kHid, kHid};
    const int offs[5] = {0, kOffW2, kOffW3, kOffW4, kParams};
    for (int layer = 0; layer < 4; ++layer) {
        const float bound = 1.0f / sqrtf((float)fan_in[layer]);
        for (int i = offs[layer]; i < offs[layer + 1]; ++i) {
            const double u = (double)(splitmix64(st) >> 11) * (1.0 / 9007199254740992.0);
            h[i] = (float)((2.0 * u - 1.0) * bound);
        }
    }
    spl_status s = spl_mlp_set_params(m, h);
    free(h);
    if (s != SPL_OK) {
        cudaFree(blk);
        free(m);
        return s;
    }
    *out = m;
    return SPL_OK;
}

extern "C" void spl_mlp_destroy(spl_mlp *m)
{
    if (!m) return;
    if (m->block) cudaFree(m->block);
    free(m);
}

extern "C" spl_status spl_mlp_set_params(spl_mlp *m, const float *host_params)
{
    clear_error();
    if (!m || !host_params) return fail(SPL_ERR_ARG, "NULL argument");
    for (int i = 0; i < kParams; ++i)
        if (!isfinite(host_params[i])) return fail(SPL_ERR_NONFINITE, "parameter %d is not finite", i);
    spl_status s = cuda_check(cudaMemcpy(m->master, host_params, kParams * 4, cudaMemcpyHostToDevice), "params upload");
    if (s != SPL_OK) return s;
    s = cuda_check(cudaMemset(m->adam_m, 0, kParams * 4), "adam reset");
    if (s != SPL_OK) return s;
    s = cuda_check(cudaMemset(m->adam_v, 0, kParams * 4), "adam reset");
    if (s != SPL_OK) return s;
    m->step = 0;
    s = prep(m, 0);
    if (s != SPL_OK) return s;
    return cuda_check(cudaDeviceSynchronize(), "params prep");
}

extern "C" spl_status spl_mlp_status(const spl_mlp *m, void *stream)
{
    clear_error();
    if (!m) return fail(SPL_ERR_ARG, "mlp is NULL");
    cudaStream_t st = (cudaStream_t)stream;
    int flag = 0;
    spl_status s = cuda_check(cudaMemcpyAsync(&flag, m->err, sizeof(int), cudaMemcpyDeviceToHost, st), "status read");
    if (s == SPL_OK) s = cuda_check(cudaStreamSynchronize(st), "status sync");
    if (s != SPL_OK) return s;
    if (flag) {
        s = cuda_check(cudaMemsetAsync(m->err, 0, sizeof(int), st), "status clear");
        if (s == SPL_OK) s = cuda_check(cudaStreamSynchronize(st), "status sync");
        if (s != SPL_OK) return s;
        return fail(SPL_ERR_TIMEOUT, "a bounded tensor-core wait gave up (flag 0x%x)", flag);
    }
    return SPL_OK;
}

// ---------------------------------------------------------------- checkpoint
namespace {
const char kCkptMagic[8] = {'S', 'P', 'L', 'M', 'L', 'P', '2', '\0'};
constexpr int kCkptVersion = 2;
constexpr int kCkptHeader = 8;  // int32 fields after the magic

void put_le32(unsigned char *b, uint32_t v)
{
    for (int i = 0; i < 4; ++i) b[i] = (unsigned char)(v >> (8 * i));
}
uint32_t get_le32(const unsigned char *b)
{
    uint32_t v = 0;
    for (int i = 0; i < 4; ++i) v |= (uint32_t)b[i] << (8 * i);
    return v;
}
}  // namespace

extern "C" spl_status spl_mlp_save(const spl_mlp *m, const char *path)
{
    clear_error();
    if (!m || !path) return fail(SPL_ERR_ARG, "NULL argument");
    const size_t nbytes = 8 + 4 * kCkptHeader + 8 + 3 * (size_t)kParams * 4;
    unsigned char *buf = (unsigned char *)malloc(nbytes);
    if (!buf) return fail(SPL_ERR_OOM, "host allocation failed");
    memcpy(buf, kCkptMagic, 8);
    const int32_t head[kCkptHeader] = {kCkptVersion, m->degree, kParams, kIn, kHid, 3, 0, m->step};
    for (int i = 0; i < kCkptHeader; ++i) put_le32(buf + 8 + 4 * i, (uint32_t)head[i]);
    unsigned char *p = buf + 8 + 4 * kCkptHeader;
    put_le32(p, (uint32_t)(m->seed & 0xffffffffu));
    put_le32(p + 4, (uint32_t)(m->seed >> 32));
    p += 8;
    float *tmp = (float *)malloc((size_t)kParams * 4);
    if (!tmp) {
        free(buf);
        return fail(SPL_ERR_OOM, "host allocation failed");
    }
    const float *src[3] = {m->master, m->adam_m, m->adam_v};
    spl_status s = cuda_check(cudaDeviceSynchronize(), "checkpoint sync");
    for (int a = 0; a < 3 && s == SPL_OK; ++a) {
        s = cuda_check(cudaMemcpy(tmp, src[a], (size_t)kParams * 4, cudaMemcpyDeviceToHost), "checkpoint download");
        for (int i = 0; i < kParams && s == SPL_OK; ++i) {
            uint32_t bits;
            memcpy(&bits, tmp + i, 4);
            put_le32(p + 4 * ((size_t)a * kParams + i), bits);
        }
    }
    free(tmp);
    if (s == SPL_OK) {
        FILE *f = fopen(path, "wb");
        if (!f) s = fail(SPL_ERR_ARG, "cannot open %s for writing", path);
        else {
            const size_t w = fwrite(buf, 1, nbytes, f);
            const int c = fclose(f);
            if (w != nbytes || c != 0) s = fail(SPL_ERR_ARG, "write to %s failed", path);
        }
    }
    free(buf);
    return s;
}

extern "C" spl_status spl_mlp_load(spl_mlp *m, const char *path)
{
    clear_error();
    if (!m || !path) return fail(SPL_ERR_ARG, "NULL argument");
    const size_t nbytes = 8 + 4 * kCkptHeader + 8 + 3 * (size_t)kParams * 4;
    FILE *f = fopen(path, "rb");
    if (!f) return fail(SPL_ERR_ARG, "cannot open %s", path);
    unsigned char *buf = (unsigned char *)malloc(nbytes + 1);
    if (!buf) {
        fclose(f);
        return fail(SPL_ERR_OOM, "host allocation failed");
    }
    const size_t got = fread(buf, 1, nbytes + 1, f);
    fclose(f);
    spl_status s = SPL_OK;
    int32_t head[kCkptHeader];
    if (got != nbytes) s = fail(SPL_ERR_ARG, "%s: %zu bytes, expected %zu", path, got, nbytes);
    else if (memcmp(buf, kCkptMagic, 8) != 0) s = fail(SPL_ERR_ARG, "%s is not an f_theta checkpoint", path);
    if (s == SPL_OK) {
        for (int i = 0; i < kCkptHeader; ++i) head[i] = (int32_t)get_le32(buf + 8 + 4 * i);
        if (head[0] != kCkptVersion || head[2] != kParams || head[3] != kIn || head[4] != kHid || head[5] != 3 ||
            head[6] != 0)
            s = fail(SPL_ERR_ARG, "%s: unsupported version or network shape", path);
        else if (head[1] != m->degree)
            s = fail(SPL_ERR_ARG, "%s holds a network for degree %d, not %d", path, head[1], m->degree);
        else if (head[7] < 0)
            s = fail(SPL_ERR_ARG, "%s: negative step count", path);
    }
    float *vals = nullptr;
    if (s == SPL_OK) {
        vals = (float *)malloc(3 * (size_t)kParams * 4);
        if (!vals) s = fail(SPL_ERR_OOM, "host allocation failed");
    }
    if (s == SPL_OK) {
        const unsigned char *p = buf + 8 + 4 * kCkptHeader + 8;
        for (size_t i = 0; i < 3 * (size_t)kParams; ++i) {
            const uint32_t bits = get_le32(p + 4 * i);
            memcpy(vals + i, &bits, 4);
            if (!isfinite(vals[i])) {
                s = fail(SPL_ERR_NONFINITE, "%s: value %zu is not finite", path, i);
                break;
            }
        }
    }
    if (s == SPL_OK) {
        const unsigned char *p = buf + 8 + 4 * kCkptHeader;
        float *dst[3] = {m->master, m->adam_m, m->adam_v};
        s = cuda_check(cudaDeviceSynchronize(), "checkpoint sync");
        for (int a = 0; a < 3 && s == SPL_OK; ++a)
            s = cuda_check(cudaMemcpy(dst[a], vals + (size_t)a * kParams, (size_t)kParams * 4, cudaMemcpyHostToDevice),
                           "checkpoint upload");
        if (s == SPL_OK) {
            m->step = head[7];
            m->seed = (unsigned long long)get_le32(p) | ((unsigned long long)get_le32(p + 4) << 32);
            s = prep(m, 0);
        }
        if (s == SPL_OK) s = cuda_check(cudaDeviceSynchronize(), "checkpoint prep");
    }
    free(vals);
    free(buf);
    return s;
}

extern "C" spl_status spl_mlp_get_params(const spl_mlp *m, float *host_params)
{
    clear_error();
    if (!m || !host_params) return fail(SPL_ERR_ARG, "NULL argument");
    return cuda_check(cudaMemcpy(host_params, m->master, kParams * 4, cudaMemcpyDeviceToHost), "params download");
}

extern "C" spl_status spl_mlp_eval(const spl_mlp *m, long long count, const float *feat_dev, float *out_dev,
                                   void *stream)
{
    clear_error();
    if (!m) return fail(SPL_ERR_ARG, "mlp is NULL");
    if (count < 0) return fail(SPL_ERR_ARG, "bad count");
    if (count == 0) return SPL_OK;
    if (!feat_dev || !out_dev) return fail(SPL_ERR_ARG, "NULL array");
    spl_status s = rows_smem_attr<false>();
    if (s != SPL_OK) return s;
    k_mlp_rows<false><<<eval_blocks(count), 2 * kTcRows, sizeof(TcMlpSmem<1>), (cudaStream_t)stream>>>(
        mlp_dev(m), m->degree, count, feat_dev, nullptr, out_dev);
    return cuda_check(cudaGetLastError(), "mlp eval launch");
}

extern "C" spl_status spl_mlp_grad(spl_mlp *m, int batch, const float *feat_dev, const float *target_dev,
                                   float *grad_dev, float *loss_dev, void *stream)
{
    clear_error();
    if (!m || !feat_dev || !target_dev || !grad_dev) return fail(SPL_ERR_ARG, "NULL argument");
    if (batch < 1 || batch > m->max_batch) return fail(SPL_ERR_ARG, "batch %d not in 1..%d", batch, m->max_batch);
    return grad_impl(m, batch, feat_dev, target_dev, grad_dev, loss_dev, (cudaStream_t)stream);
}

extern "C" spl_status spl_mlp_train_step(spl_mlp *m, int batch, const float *feat_dev, const float *target_dev,
                                         float lr, float *loss_dev, void *stream)
{
    clear_error();
    if (!m || !feat_dev || !target_dev) return fail(SPL_ERR_ARG, "NULL argument");
    if (batch < 1 || batch > m->max_batch) return fail(SPL_ERR_ARG, "batch %d not in 1..%d", batch, m->max_batch);
    if (!(lr >= 0.0f) || !isfinite(lr)) return fail(SPL_ERR_ARG, "bad learning rate");
    cudaStream_t st = (cudaStream_t)stream;
    spl_status s = grad_impl(m, batch, feat_dev, target_dev, m->grad, loss_dev, st);
    if (s != SPL_OK) return s;
    m->step += 1;
    const float c1 = 1.0f - powf(0.9f, (float)m->step), c2 = 1.0f - powf(0.999f, (float)m->step);
    k_adam<<<(kParams + 255) / 256, 256, 0, st>>>(m->master, m->adam_m, m->adam_v, m->grad, lr, c1, c2);
    s = cuda_check(cudaGetLastError(), "adam launch");
    if (s != SPL_OK) return s;
    return prep(m, st);
}
