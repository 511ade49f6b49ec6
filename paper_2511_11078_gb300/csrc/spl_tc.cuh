// spl_tc.cuh -- the learned footprint f_theta (Sec. 2.2) on the 5th-generation
// tensor cores: tcgen05.mma with operands in shared memory and the FP32
// accumulator in tensor memory (TMEM).
//
// A group of 128 or 256 threads (a CTA, or a part of one) evaluates tiles of
// 128 rows, with one thread per row or two (each taking half of the row's 64
// columns).  Each layer is one M=128 x N=64 product: the threads write their
// parts of the A operand (BF16) to shared memory, one thread issues the MMAs,
// the tensor core accumulates the 128 x 64 FP32 result in 64 TMEM columns,
// and every thread reads its part back with tcgen05.ld (TMEM lane = row),
// applies SiLU and writes the next layer's A operand.  The MMAs take no issue
// slots of the other threads and no registers: what is left to the threads is
// SiLU, the BF16 packing and the 64 -> 1 output layer.  A layer's barrier,
// MMA and TMEM round trip are hidden by the other groups of the SM.
//
// Precision contract (the one the oracle emulates): layers 2 and 3 multiply
// BF16 weights with the BF16-rounded activations, accumulating in FP32;
// layer 1 and the biases keep FP32 accuracy through three-part BF16 splits
// x = hi + mid + lo (hi and mid truncate the mantissa to 8 bits, the
// differences being exact in FP32; lo rounds the remainder to nearest, so
// what is dropped is below 2^-23 |x|): layer 1 multiplies
// [hi(x), mid(x), lo(x), 0] (16 columns) with [W1; W1; W1; 0], and each
// bias enters through one more K=16 step whose A rows are (1, 1, 1, 0 ...)
// and whose B rows are (hi(b), mid(b), lo(b), 0 ...).  The output layer is
// FP32 on the CUDA cores.
//
// Operand layout: the canonical K-major layout without swizzling.  An
// operand of R rows and K columns (BF16) is made of 8-row x 16-byte core
// matrices; core matrix (row group i, column group j) sits at byte
// j * (R / 8) * 128 + i * 128, row r of it at + 16 r.  The shared-memory
// descriptor takes the distance between core matrices along K (leading
// byte offset, (R / 8) * 128) and along the rows (stride byte offset, 128).
#pragma once

#include <stddef.h>

#include "spl_mlp.cuh"

namespace spl {
namespace tc {

__device__ __forceinline__ uint32_t saddr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// Shared-memory matrix descriptor (tcgen05 format): start address, leading
// and stride byte offsets (all in 16-byte units), descriptor version 1 at
// bit 46, base offset 0, no swizzling.
__device__ __forceinline__ uint64_t desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), A
// and B BF16 (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 = 0),
// N / 8 at bits 17-22, M / 16 at bits 24-28.
constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D (TMEM) = A * B (+ D when acc), A and B from shared memory
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

// arrive on the mbarrier once every MMA this thread issued so far is complete
__device__ __forceinline__ void commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(bar))
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count) : "memory");
}

// Wait for the phase with the given parity to complete; gives up (false)
// after a bounded number of polls.
constexpr unsigned kWaitPolls = 1u << 20;
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity, unsigned polls = kWaitPolls)
{
    const uint32_t a = saddr(bar);
    for (unsigned it = 0; it < polls; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// barrier over `threads` threads (a group of the CTA's warps), reached by
// each thread on its own (not .aligned)
__device__ __forceinline__ void bar_sync(int id, int threads)
{
    asm volatile("barrier.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// make this thread's generic-proxy shared-memory writes visible to the
// tensor core (async proxy)
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// warp-wide: allocate ncols TMEM columns, base address written to *dst
__device__ __forceinline__ void alloc(uint32_t *dst, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(saddr(dst)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// 32 consecutive FP32 columns of the warp's 32 TMEM lanes (lane = thread)
// into v[O .. O + 31]
template <int O, int L>
__device__ __forceinline__ void ld32(uint32_t taddr, float (&v)[L])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 32; ++i) v[O + i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

}  // namespace tc

constexpr int kTcRows = 128;  // rows of a tile
constexpr int kTcCols = 64;   // TMEM columns of the accumulator (N = 64, FP32)

// The network in the tile's operand layout (built once per parameter
// update in global memory, copied into every CTA's shared memory).
struct __align__(16) TcMlpImage {
    uint8_t w2[64 * 64 * 2];        // B of layer 2: 64 (N) x 64 (K)
    uint8_t w3[64 * 64 * 2];
    uint8_t w1[64 * 16 * 2];        // B of layer 1: 64 x 16, [W1; W1; W1; 0]
    uint8_t bias[3][64 * 16 * 2];   // B of the bias steps of layers 1-3
    uint8_t one[kTcRows * 16 * 2];  // A of the bias steps: rows (1, 1, 1, 0 ...)
    float w4[64];
    float b4;
    float pad[3];
};

// A group's operands: A of layers 2 and 3 (128 x 64), whose first 4 KB also
// hold A of layer 1 (128 x 16; read before layer 2's is written).
struct __align__(128) TcTile {
    uint8_t a2[kTcRows * 64 * 2];
    uint32_t tmem;   // the group's 64 accumulator columns
    int stop;        // a completion wait of the group gave up
    uint64_t mbar;
};
// Shared memory of a CTA: the network image and one tile per group.
template <int GROUPS> struct __align__(1024) TcMlpSmem {
    TcMlpImage img;
    TcTile tile[GROUPS];
};

static_assert(sizeof(TcMlpImage) % 16 == 0, "the image is copied in 16-byte units");
static_assert(offsetof(TcMlpSmem<2>, tile) % 16 == 0 && sizeof(TcTile) % 16 == 0,
              "operands start on 16-byte boundaries (shared-memory descriptors)");
// TMEM allocation never waits: a CTA holds at least sizeof(TcMlpSmem<GROUPS>)
// of shared memory for 64 GROUPS columns, so the CTAs of an SM (228 KB) stay
// below its 512 columns.
template <int GROUPS> constexpr size_t tc_max_cols()
{
    return 228 * 1024 / (sizeof(TcMlpSmem<GROUPS>) + 1024) * (kTcCols * GROUPS);
}
static_assert(tc_max_cols<1>() <= 512 && tc_max_cols<2>() <= 512, "TMEM columns of the CTAs an SM can hold");

// byte offset of element (row, k) in an operand of R rows (K-major, no swizzle)
__host__ __device__ constexpr uint32_t kmaj_off(int R, int row, int k)
{
    return (uint32_t)((k >> 3) * (R / 8) * 128 + (row >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint16_t bf16_bits_rn(float x)
{
    __nv_bfloat16 h = __float2bfloat16_rn(x);
    return *reinterpret_cast<uint16_t *>(&h);
}
// three-part split of an FP32 value (hi, mid truncated, lo rounded)
__device__ __forceinline__ void split3(float x, uint16_t &hi, uint16_t &mid, uint16_t &lo)
{
    const uint32_t bx = __float_as_uint(x);
    const float r1 = x - __uint_as_float(bx & 0xFFFF0000u);
    const uint32_t b1 = __float_as_uint(r1);
    const float r2 = r1 - __uint_as_float(b1 & 0xFFFF0000u);
    hi = (uint16_t)(bx >> 16);
    mid = (uint16_t)(b1 >> 16);
    lo = bf16_bits_rn(r2);
}

// The network image from the FP32 parameter vector P (layout kOff*): the
// same BF16 roundings as the evaluation copy (W1, W2, W3, W4 rounded to
// nearest BF16, the biases split, b4 unrounded); grid-stride over the
// calling threads (tid of nthreads).
__device__ __forceinline__ void tc_mlp_image(const float *__restrict__ P, TcMlpImage &I, int tid, int nthreads)
{
    uint16_t *w1 = reinterpret_cast<uint16_t *>(I.w1);
    for (int i = tid; i < 64 * 16; i += nthreads) {
        const int n = i >> 4, k = i & 15;
        w1[kmaj_off(64, n, k) / 2] = bf16_bits_rn(k < 15 ? P[kOffW1 + n * kIn + k % 5] : 0.0f);
    }
    // hidden layers: 16-byte units (row n, columns 8j .. 8j+7)
    for (int i = tid; i < 2 * 64 * 8; i += nthreads) {
        const int layer = i >> 9, n = (i >> 3) & 63, j = i & 7;
        const float *W = P + (layer == 0 ? kOffW2 : kOffW3) + n * kHid + 8 * j;
        const uint4 v = make_uint4(pack_bf16(W[0], W[1]), pack_bf16(W[2], W[3]), pack_bf16(W[4], W[5]),
                                   pack_bf16(W[6], W[7]));
        *reinterpret_cast<uint4 *>((layer == 0 ? I.w2 : I.w3) + kmaj_off(64, n, 8 * j)) = v;
    }
    for (int i = tid; i < 3 * 64 * 16; i += nthreads) {
        const int layer = i >> 10, n = (i >> 4) & 63, k = i & 15;
        uint16_t hi, mid, lo;
        split3(P[(layer == 0 ? kOffB1 : (layer == 1 ? kOffB2 : kOffB3)) + n], hi, mid, lo);
        const uint16_t v = k == 0 ? hi : (k == 1 ? mid : (k == 2 ? lo : (uint16_t)0));
        reinterpret_cast<uint16_t *>(I.bias[layer])[kmaj_off(64, n, k) / 2] = v;
    }
    for (int i = tid; i < kTcRows * 16; i += nthreads) {
        const int m = i >> 4, k = i & 15;
        reinterpret_cast<uint16_t *>(I.one)[kmaj_off(kTcRows, m, k) / 2] = k < 3 ? (uint16_t)0x3F80u : (uint16_t)0;
    }
    for (int i = tid; i < 64; i += nthreads) I.w4[i] = __bfloat162float(__float2bfloat16_rn(P[kOffW4 + i]));
    if (tid == 0) {
        I.b4 = P[kOffB4];
        I.pad[0] = I.pad[1] = I.pad[2] = 0.0f;
    }
}

// The network image into shared memory (16-byte copies), the groups'
// completion barriers and TMEM accumulators.  Called by all threads of the
// CTA; ends with a CTA barrier.
template <int GROUPS>
__device__ __forceinline__ void tc_mlp_setup(const MlpDev &w, TcMlpSmem<GROUPS> &S)
{
    const int tid = threadIdx.x;
    const uint4 *src = reinterpret_cast<const uint4 *>(w.tc_img);
    uint4 *dst = reinterpret_cast<uint4 *>(&S.img);
    for (int i = tid; i < (int)(sizeof(TcMlpImage) / 16); i += blockDim.x) dst[i] = __ldg(src + i);
    if (tid == 0) {
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) {
            tc::mbar_init(&S.tile[g].mbar, 1);
            S.tile[g].stop = 0;
        }
        tc::fence_mbar_init();
    }
    if (tid < 32) {
        __syncwarp();  // lane 0 comes from a branch of its own, the allocation is warp-wide
        tc::alloc(&S.tile[0].tmem, kTcCols * GROUPS);
    }
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (GROUPS > 1) {
        if (tid == 0)
#pragma unroll
            for (int g = 1; g < GROUPS; ++g) S.tile[g].tmem = S.tile[0].tmem + (uint32_t)(g * kTcCols);
        __syncthreads();
    }
}

// Release the TMEM accumulators.  Called by all threads of the CTA.  When a
// completion wait gave up (`pending`), the group's last committed MMAs may
// still be running: wait once more, bounded, for the phase of the last commit
// (`phase` is the parity the next wait would use) before the columns are
// freed.
template <int GROUPS>
__device__ __forceinline__ void tc_mlp_teardown(TcMlpSmem<GROUPS> &S, TcTile &T, unsigned phase = 0u, bool pending = false)
{
    if (pending) tc::mbar_wait(&T.mbar, phase ^ 1u);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (threadIdx.x < 32) tc::dealloc(S.tile[0].tmem, kTcCols * GROUPS);
}

// One MMA layer: D = sum over k-steps of A * B, plus the bias step; the
// group's thread `tid` 0 issues, everyone waits for completion (a group that
// has given up before does not wait again).  nk: K=16 steps of the A operand
// (A columns 16 s .. 16 s + 15 at a + s * (rows / 8) * 256 bytes, B at
// b + s * 8 * 256).  bar: the group's barrier, of `threads` threads.
__device__ __forceinline__ bool tc_layer(const TcMlpImage &img, TcTile &T, int tid, int bar, int threads, const uint8_t *b,
                                         int nk, int layer, unsigned &phase, bool ok)
{
    constexpr uint32_t idesc = tc::idesc_bf16(kTcRows, 64);
    tc::fence_proxy_async();
    tc::fence_before();
    tc::bar_sync(bar, threads);
    if (tid == 0) {
        tc::fence_after();
        const uint32_t sa = tc::saddr(T.a2), sb = tc::saddr(b);
        for (int s = 0; s < nk; ++s)
            tc::mma(T.tmem, tc::desc(sa + s * (kTcRows / 8) * 256, (kTcRows / 8) * 128, 128),
                    tc::desc(sb + s * 8 * 256, 8 * 128, 128), idesc, s > 0);
        tc::mma(T.tmem, tc::desc(tc::saddr(img.one), (kTcRows / 8) * 128, 128),
                tc::desc(tc::saddr(img.bias[layer]), 8 * 128, 128), idesc, 1);
        tc::commit(&T.mbar);
    }
    ok = tc::mbar_wait(&T.mbar, phase, ok ? tc::kWaitPolls : 1u) && ok;
    phase ^= 1u;
    tc::fence_after();
    return ok;
}

// Threads per row of a tile: TPR = 1 (128 threads, a whole row each) or
// TPR = 2 (256 threads; warps w and w + 4 read the same TMEM lane quarter,
// w % 4, and take columns 0..31 and 32..63 of its rows): half the serial
// work per thread, for batches too small to fill the GPU with 128-row tiles.
// (threadIdx.x & 96 is the warp's TMEM lane quarter, 32 * (warp % 4).)

// Columns C0 .. C0 + 31 of this thread's row of the accumulator.  tcgen05.ld is
// warp-wide, and the lanes may come apart before it: in the completion wait,
// and where only some of them repeat their SiLU values (tc_silu_store).
template <int C0>
__device__ __forceinline__ void tc_cols(uint32_t tmem, float (&z)[32])
{
    __syncwarp();
    tc::ld32<0>(tmem + ((uint32_t)(threadIdx.x & 96) << 16) + (uint32_t)C0, z);
    tc::wait_ld();
}

// SiLU of four values, z / d with d = 1 + 2^(-z log2 e), through one MUFU
// reciprocal of the four denominators' product instead of one each: with
// P = (d0 d2, d1 d3) and r = 1 / (P.x P.y), 1 / d0 = (r P.y) d2 and so on.
// GB300's MUFU takes base-2 exponentials at twice the rate of reciprocals, so
// a reciprocal per value was two thirds of its work (a quarter of them by
// Newton steps on the FMA pipe); now it is a fifth.  Each reciprocal carries
// four more roundings of 2^-24 than rcp(d) itself, far below the BF16 rounding
// that follows in the hidden layers; the output layer, which is FP32, keeps a
// reciprocal for each value (silu2; a view of the 256^3 cone 32.3 -> 33.4 ms,
// A^T 32.0 -> 32.6; the shared one with a residual step 33.9 and 33.3).  Values
// below -87 can take the product out of range (`over`
// collects the largest; the caller then repeats its values with silu_safe).
__device__ __forceinline__ void silu4(const float (&z)[4], float (&h)[4], float &over)
{
    constexpr float kNegLog2e = -1.4426950408889634f;
    const float2 one = make_float2(1.0f, 1.0f), k = make_float2(kNegLog2e, kNegLog2e);
    const float2 za = make_float2(z[0], z[1]), zb = make_float2(z[2], z[3]);
    const float2 ma = __fmul2_rn(za, k), mb = __fmul2_rn(zb, k);
    const float2 da = __fadd2_rn(make_float2(ex2_approx(ma.x), ex2_approx(ma.y)), one);
    const float2 db = __fadd2_rn(make_float2(ex2_approx(mb.x), ex2_approx(mb.y)), one);
    const float2 P = __fmul2_rn(da, db);
    const float q = P.x * P.y, r = rcp_approx(q);
    over = fmaxf(over, q);
    const float2 R = make_float2(r * P.y, r * P.x);
    const float2 ha = __fmul2_rn(za, __fmul2_rn(R, db)), hb = __fmul2_rn(zb, __fmul2_rn(R, da));
    h[0] = ha.x;
    h[1] = ha.y;
    h[2] = hb.x;
    h[3] = hb.y;
}
constexpr float kSiluOver = 0x1p125f;  // above it the reciprocal is not a normal number
// one value at a time; d is capped where SiLU is below 1e-36 either way
__device__ __forceinline__ float silu_safe(float z)
{
    return z * rcp_approx(fminf(1.0f + ex2_approx(-1.4426950408889634f * z), 0x1p126f));
}

// SiLU of 32 columns of a row from column c0, rounded to BF16 into the row of
// the A operand of the next layer (and, with SAVE, z and the rounded
// activations to zb / hb, which point at the row).
template <bool SAVE>
__device__ __forceinline__ void tc_silu_store(TcTile &T, int m, int c0, const float (&z)[32], float *zb, float *hb)
{
    if (SAVE) {
#pragma unroll
        for (int k = 0; k < 32; k += 4)
            *reinterpret_cast<float4 *>(zb + c0 + k) = make_float4(z[k], z[k + 1], z[k + 2], z[k + 3]);
    }
    float over = 0.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float zz[4] = {z[8 * j + 4 * q], z[8 * j + 4 * q + 1], z[8 * j + 4 * q + 2], z[8 * j + 4 * q + 3]};
            float h[4];
            silu4(zz, h, over);
            w[2 * q] = pack_bf16(h[0], h[1]);
            w[2 * q + 1] = pack_bf16(h[2], h[3]);
        }
        *reinterpret_cast<uint4 *>(T.a2 + kmaj_off(kTcRows, m, c0 + 8 * j)) = make_uint4(w[0], w[1], w[2], w[3]);
        if (SAVE) {
            float4 *d = reinterpret_cast<float4 *>(hb + c0 + 8 * j);
            d[0] = make_float4(__uint_as_float(w[0] << 16), __uint_as_float(w[0] & 0xFFFF0000u),
                               __uint_as_float(w[1] << 16), __uint_as_float(w[1] & 0xFFFF0000u));
            d[1] = make_float4(__uint_as_float(w[2] << 16), __uint_as_float(w[2] & 0xFFFF0000u),
                               __uint_as_float(w[3] << 16), __uint_as_float(w[3] & 0xFFFF0000u));
        }
    }
    if (over > kSiluOver) {
        // some value far below zero: again, one by one
#pragma unroll 1
        for (int c = 0; c < 32; ++c) {
            float v = z[0];
#pragma unroll
            for (int e = 1; e < 32; ++e) v = e == c ? z[e] : v;
            const uint16_t b = bf16_bits_rn(silu_safe(v));
            *reinterpret_cast<uint16_t *>(T.a2 + kmaj_off(kTcRows, m, c0 + c)) = b;
            if (SAVE) hb[c0 + c] = __uint_as_float((uint32_t)b << 16);
        }
    }
}

// Optional capture of a tile's activations for training: z1, h1, z2, h2,
// z3, h3 of this thread's row (FP32; h1, h2 as the BF16-rounded values that
// entered the tensor-core layers), 64 values each at row * 64 of the arrays
// (row < 0: nothing is stored).
struct TcSave {
    float *z1, *h1, *z2, *h2, *z3, *h3;
    int row;
};

// Output layer over 32 columns of a row from column c0: o += w4 . SiLU(z).
template <bool SAVE>
__device__ __forceinline__ float tc_output(const TcMlpImage &img, int c0, const float (&z)[32], bool save, float *zb, float *hb)
{
    float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
        if (SAVE && save) *reinterpret_cast<float4 *>(zb + c0 + k) = make_float4(z[k], z[k + 1], z[k + 2], z[k + 3]);
        const float2 h0 = silu2(make_float2(z[k], z[k + 1])), h1 = silu2(make_float2(z[k + 2], z[k + 3]));
        if (SAVE && save) *reinterpret_cast<float4 *>(hb + c0 + k) = make_float4(h0.x, h0.y, h1.x, h1.y);
        const float4 w = *reinterpret_cast<const float4 *>(img.w4 + c0 + k);
        acc = __ffma2_rn(h0, make_float2(w.x, w.y), acc);
        acc = __ffma2_rn(h1, make_float2(w.z, w.w), acc);
    }
    return acc.x + acc.y;
}

// f_theta of this thread's row x (5 features) in a tile of 128 rows; every
// thread of the group (128 * TPR; `tid` its number in the group, `bar` the
// group's barrier) calls it, the TPR threads of a row with the same x.
// Returns false if a tensor-core wait gave up, now or before (`ok`; the output
// is then meaningless).  The output is valid in every thread of the row.
// part: 2 x 128 floats of shared memory for combining the halves of the output
// layer (TPR = 2; rewritten only after the next tile's first barrier).
// SAVE stores the activations of the row (sv->row >= 0).
template <int TPR, bool SAVE = false>
__device__ __forceinline__ bool tc_mlp_tile(const TcMlpImage &img, TcTile &T, int tid, int bar, bool ok, const float (&x)[5],
                                            float &out, unsigned &phase, float *part = nullptr, const TcSave *sv = nullptr)
{
    constexpr int threads = kTcRows * TPR;
    const int m = tid & (kTcRows - 1), half = TPR == 1 ? 0 : tid >> 7;
    const bool save = SAVE && sv->row >= 0;
    const size_t ro = SAVE ? (size_t)(sv->row < 0 ? 0 : sv->row) * 64 : 0;
    {
        uint16_t p[16];
#pragma unroll
        for (int e = 0; e < 5; ++e) split3(x[e], p[e], p[5 + e], p[10 + e]);
        p[15] = 0;
        uint32_t v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = (uint32_t)p[2 * q] | ((uint32_t)p[2 * q + 1] << 16);
        if (TPR == 1 || half == 0)
            *reinterpret_cast<uint4 *>(T.a2 + kmaj_off(kTcRows, m, 0)) = make_uint4(v[0], v[1], v[2], v[3]);
        if (TPR == 1 || half == 1)
            *reinterpret_cast<uint4 *>(T.a2 + kmaj_off(kTcRows, m, 8)) = make_uint4(v[4], v[5], v[6], v[7]);
    }
    const uint32_t tm = T.tmem;
    // 32 columns at a time: 32 values in registers instead of 64
    auto hidden = [&](float *zb, float *hb) {
        float z[32];
        auto store = [&](int c0) {
            if (save) tc_silu_store<true>(T, m, c0, z, zb + ro, hb + ro);
            else tc_silu_store<false>(T, m, c0, z, nullptr, nullptr);
        };
        if (TPR == 1 || half == 0) {
            tc_cols<0>(tm, z);
            store(0);
        }
        if (TPR == 1 || half == 1) {
            tc_cols<32>(tm, z);
            store(32);
        }
    };
    ok = tc_layer(img, T, tid, bar, threads, img.w1, 1, 0, phase, ok);
    hidden(SAVE ? sv->z1 : nullptr, SAVE ? sv->h1 : nullptr);
    ok = tc_layer(img, T, tid, bar, threads, img.w2, 4, 1, phase, ok);
    hidden(SAVE ? sv->z2 : nullptr, SAVE ? sv->h2 : nullptr);
    ok = tc_layer(img, T, tid, bar, threads, img.w3, 4, 2, phase, ok);
    float o = 0.0f;
    {
        float z[32];
        float *zb = SAVE ? sv->z3 + ro : nullptr, *hb = SAVE ? sv->h3 + ro : nullptr;
        if (TPR == 1 || half == 0) {
            tc_cols<0>(tm, z);
            o = tc_output<SAVE>(img, 0, z, save, zb, hb);
        }
        if (TPR == 1 || half == 1) {
            tc_cols<32>(tm, z);
            o += tc_output<SAVE>(img, 32, z, save, zb, hb);
        }
    }
    if (TPR == 2) {
        // both threads of the row add the two halves in the same order
        part[half * kTcRows + m] = o;
        tc::bar_sync(bar, threads);
        o = part[m] + part[kTcRows + m];
    }
    out = o + img.b4;
    return ok;
}

}  // namespace spl
