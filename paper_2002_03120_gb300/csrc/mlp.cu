// mlp.cu -- the apparent-viscosity surrogate network on GB300 tensor cores.
//
// Network (a build component, not in the paper): 3 -> 128 -> 128 -> 128 ->
// 128 -> 1, GELU (erf form) after every hidden layer, MSE loss, Adam.  The
// three 128 x 128 layers run as tcgen05 MMAs (kind::f16, BF16 operands for
// both A and B, FP32 accumulators in tensor memory); the 3 -> 128 input layer,
// the 128 -> 1 output layer and all element-wise work run in FP32 on the CUDA
// cores.  One MMA tile is M = 128 rows x N = 128 x K = 128 (eight K = 16
// steps), issued by one thread; completion is signalled through an mbarrier
// by tcgen05.commit; the epilogue reads the accumulator rows with tcgen05.ld
// (thread t of the 128 owns row t = TMEM lane t).
//
// Shared-memory operands use the canonical K-major layout without swizzle:
// 8-row x 16-byte core matrices, core (row group g, K chunk c) at byte offset
// (16 g + c) * 128 of a 32 KB tile; descriptor leading-dimension offset 128 B
// (next K chunk), stride-dimension offset 2048 B (next 8-row group).  Every
// address an MMA can touch lies inside its 32 KB tile.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include <cuda_bf16.h>

#include "common.cuh"

namespace sdpd {
namespace mlp {

constexpr int WID = 128;
constexpr int NIN = 3;
constexpr int TILE_BYTES = WID * WID * 2;  // one 128 x 128 bf16 operand
constexpr int NPARAM = WID * NIN + WID + 3 * (WID * WID + WID) + WID + 1;
// flat parameter offsets: W0 [128][3], b0, W1 [128][128], b1, W2, b2, W3, b3, W4 [128], b4
constexpr int OFF_W0 = 0, OFF_B0 = OFF_W0 + WID * NIN;
__host__ __device__ constexpr int off_W(int l) { return OFF_B0 + WID + (l - 1) * (WID * WID + WID); }
__host__ __device__ constexpr int off_b(int l) { return off_W(l) + WID * WID; }
constexpr int OFF_W4 = OFF_B0 + WID + 3 * (WID * WID + WID), OFF_B4 = OFF_W4 + WID;
static_assert(OFF_B4 + 1 == NPARAM, "parameter layout");
// one tile's gradient share: padded so that every share starts on 16 bytes
constexpr int GSTRIDE = (NPARAM + 3) / 4 * 4;
static_assert((NPARAM + 255) / 256 * 256 > NPARAM, "the reduction has a thread past the parameters for the loss");
static_assert(off_W(1) % 4 == 0 && (WID * WID + WID) % 4 == 0, "weight gradients are stored as float4");

// instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A BF16 (bits
// 7-9 = 1), B BF16 (bits 10-12 = 1), both K-major, N >> 3 at bits 17-22,
// M >> 4 at bits 24-28
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(WID >> 3) << 17) |
                           ((uint32_t)(WID >> 4) << 24);
constexpr long long WAIT_LIMIT = 1LL << 22;   // bounded mbarrier wait (iterations)
constexpr int ERR_MMA_TIMEOUT = 1;

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// byte offset of element (r, k) of a 128 x 128 operand in the core-matrix layout
__device__ __forceinline__ uint32_t core_off(int r, int k)
{
    return (uint32_t)(((r >> 3) * 16 + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ uint64_t make_desc(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)(128u >> 4) << 16;    // leading dimension byte offset: next K chunk
    d |= (uint64_t)(2048u >> 4) << 32;   // stride dimension byte offset: next 8-row group
    d |= (uint64_t)1 << 46;              // descriptor version
    return d;                            // base offset 0, no swizzle
}

__device__ __forceinline__ void tc_alloc(uint32_t *slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

__device__ __forceinline__ void tc_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mma_bf16(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, int accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(IDESC), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t *mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t *mbar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar)));
}

// Bounded wait for the phase with parity `par`; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t par)
{
    const uint32_t a = smem_u32(mbar);
    for (long long it = 0; it < WAIT_LIMIT; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, P;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(par)
            : "memory");
        if (done) return true;
    }
    return false;
}

// 16 consecutive accumulator columns of this thread's lane (row).
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float v[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// exp2 on the special-function unit (relative error about 2^-22)
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// erf by Abramowitz & Stegun, Handbook of Mathematical Functions, formula
// 7.1.26 (Hastings' rational approximation), |error| <= 1.5e-7: one
// reciprocal, one exponential, no branch.
__device__ __forceinline__ float erf_as(float x)
{
    const float a = fabsf(x);
    const float t = __fdividef(1.0f, fmaf(0.3275911f, a, 1.0f));
    float p = fmaf(1.061405429f, t, -1.453152027f);
    p = fmaf(p, t, 1.421413741f);
    p = fmaf(p, t, -0.284496736f);
    p = fmaf(p, t, 0.254829592f);
    p *= t;
    const float r = fmaf(-p, ex2_approx(-a * a * 1.44269504088896341f), 1.0f);
    return copysignf(r, x);
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// GELU, erf form: 0.5 z (1 + erf(z / sqrt 2)) = z (1 - h) for z >= 0 and
// z h for z < 0, with h = 0.5 erfc(|z| / sqrt 2) = 0.5 P(t) exp(-z^2 / 2) from
// the same Abramowitz & Stegun 7.1.26 polynomial (coefficients halved).
__device__ __forceinline__ float gelu(float z)
{
    const float a = fabsf(z) * 0.70710678118654752f;
    const float t = rcp_approx(fmaf(0.3275911f, a, 1.0f));
    float p = fmaf(0.5f * 1.061405429f, t, 0.5f * -1.453152027f);
    p = fmaf(p, t, 0.5f * 1.421413741f);
    p = fmaf(p, t, 0.5f * -0.284496736f);
    p = fmaf(p, t, 0.5f * 0.254829592f);
    const float h = (p * t) * ex2_approx(z * z * -0.72134752044448170f);
    return z * (z >= 0.0f ? 1.0f - h : h);
}
// The same operations on two values at once (packed FP32 instructions; the
// special-function unit takes one value each): the same bits.
__device__ __forceinline__ F2 gelu2(F2 z)
{
    float z0, z1, d0, d1, e0, e1;
    z.get(z0, z1);
    // (a scalar product takes the absolute value with it; the packed one would
    // cost two masks more: 10^6 rows 312 -> 303 us)
    const F2 a(fabsf(z0) * 0.70710678118654752f, fabsf(z1) * 0.70710678118654752f);
    fma2(F2(0.3275911f), a, F2(1.0f)).get(d0, d1);
    mul2(mul2(z, z), F2(-0.72134752044448170f)).get(e0, e1);
    const F2 t(rcp_approx(d0), rcp_approx(d1));
    F2 p = fma2(F2(0.5f * 1.061405429f), t, F2(0.5f * -1.453152027f));
    p = fma2(p, t, F2(0.5f * 1.421413741f));
    p = fma2(p, t, F2(0.5f * -0.284496736f));
    p = mul2(fma2(p, t, F2(0.5f * 0.254829592f)), t);
    const F2 e(ex2_approx(e0), ex2_approx(e1)), h = mul2(p, e);
    float h0, h1, g0, g1;
    h.get(h0, h1);
    fma2(h, F2(-1.0f), F2(1.0f)).get(g0, g1);
    return mul2(z, F2(z0 >= 0.0f ? g0 : h0, z1 >= 0.0f ? g1 : h1));
}
__device__ __forceinline__ float gelu_prime(float z)
{
    return 0.5f * (1.0f + erf_as(z * 0.70710678118654752f)) +
           z * ex2_approx(-0.5f * 1.44269504088896341f * z * z) * 0.39894228040143268f;
}

// Eight values of one row, written as one 16-byte core-matrix row.
__device__ __forceinline__ void put8(uint8_t *tile, int r, int k0, const F2 *v)
{
    __nv_bfloat162 h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float a, b;
        v[i].get(a, b);
        h[i] = __floats2bfloat162_rn(a, b);
    }
    *reinterpret_cast<uint4 *>(tile + core_off(r, k0)) = *reinterpret_cast<uint4 *>(h);
}

struct Net {
    float *P;            // FP32 master parameters [NPARAM]
    float *G;            // gradients [NPARAM]
    float *M, *V;        // Adam moments
    __nv_bfloat16 *Wb;   // BF16 copies of W1..W3 [3][128][128]
    float *Gp, *Lp;      // per-tile gradient shares [tiles][GSTRIDE] and squared-error sums
    float *loss;
    int *err;
    int bmax;
    long long step;
    cudaStream_t own;
};

// ------------------------------------------------------------- inference
// Persistent over 128-row tiles with NWG groups of two warpgroups per CTA:
// each group owns one tile at a time (its own activation operand in shared
// memory and its own 128 accumulator columns in tensor memory) and
// synchronises only with itself (named barrier g + 1), so the MMAs of one
// group overlap the GELU epilogues of the others.  Thread (part, row) takes
// half the columns of its row.  The three hidden weight tiles are staged once
// per CTA and shared.
// Bound by the FP32 pipe (12 packed operations for two GELUs, busy 65 % of the
// time) and by issue slots (66 %); the special-function unit is a third busy.
// 10^6 rows, calls back to back: 358 us with scalar GELUs and one thread a row,
// 303 us with packed ones, two threads a row (eight warps a scheduler instead of
// four) and the scalar absolute value.  Tiles go round the CTAs before a CTA
// gets a second one: 20,000 rows take 25 us, and took half as long again when a
// CTA was filled first.
constexpr int NWG = 4, PARTS = 2, FWD_GROUP = 128 * PARTS;
// weight and activation tiles; mbarriers, flags, TMEM slot; the input layer's
// weights and biases of two units each as pairs
constexpr size_t FWD_BARS = (size_t)(3 + NWG) * TILE_BYTES, FWD_IN = FWD_BARS + 128, FWD_SMEM = FWD_IN + (WID / 2) * 32;

__device__ __forceinline__ void wg_bar(int g) { asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(FWD_GROUP) : "memory"); }

// Row r (output unit) of one hidden weight tile, as the B operand.
__device__ __forceinline__ void stage_row(uint8_t *tile, const __nv_bfloat16 *W, int r)
{
    const uint4 *src = reinterpret_cast<const uint4 *>(W + r * WID);
#pragma unroll
    for (int c = 0; c < 16; ++c) *reinterpret_cast<uint4 *>(tile + core_off(r, 8 * c)) = __ldg(src + c);
}

// D(128 x 128) = A . B^T for warpgroup g; thread tt == 0 of the warpgroup
// issues, all 128 threads wait.  A timeout in any thread is seen by all
// (flag in shared memory read after the barrier), so the warpgroup leaves
// its loop together.
__device__ bool wg_gemm(uint8_t *A, uint8_t *B, uint32_t dtmem, uint64_t *mbar, uint32_t &parity, int g,
                        bool first, volatile int *flag, int *err)
{
    proxy_fence();
    tc_fence_before();
    wg_bar(g);
    if (first) {
        tc_fence_after();
        const uint32_t a0 = smem_u32(A), b0 = smem_u32(B);
#pragma unroll
        for (int s = 0; s < 8; ++s) mma_bf16(dtmem, make_desc(a0 + s * 256), make_desc(b0 + s * 256), s > 0 ? 1 : 0);
        mma_commit(mbar);
    }
    if (!mbar_wait(mbar, parity)) {
        *flag = 1;
        atomicOr(err, ERR_MMA_TIMEOUT);
        (void)mbar_wait(mbar, parity);
    }
    parity ^= 1u;
    tc_fence_after();
    wg_bar(g);
    return *flag == 0;
}

__global__ void __launch_bounds__(FWD_GROUP *NWG, 1) k_mlp_forward(const float *__restrict__ P,
                                                              const __nv_bfloat16 *__restrict__ Wb,
                                                              const float *__restrict__ X, float *__restrict__ Y,
                                                              long long n, int *err)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *sB = smem;                                        // 3 weight tiles
    const int g = threadIdx.x / FWD_GROUP, part = (threadIdx.x >> 7) % PARTS, tt = threadIdx.x & 127;
    const bool first = threadIdx.x % FWD_GROUP == 0;
    uint8_t *sA = smem + (3 + g) * TILE_BYTES;                 // this warpgroup's activations
    uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + (3 + NWG) * TILE_BYTES) + g;
    volatile int *flag = reinterpret_cast<int *>(smem + (3 + NWG) * TILE_BYTES + 64) + g;
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + (3 + NWG) * TILE_BYTES + 96);
    for (int r = threadIdx.x; r < 3 * WID; r += blockDim.x)
        stage_row(sB + (r >> 7) * TILE_BYTES, Wb + (r >> 7) * WID * WID, r & 127);
    float2 *sin = reinterpret_cast<float2 *>(smem + FWD_IN);   // [64][w0, w1, w2, b] of units 2i, 2i + 1
    if (threadIdx.x < WID / 2 * 4) {
        const int i = threadIdx.x >> 2, k = threadIdx.x & 3;
        sin[threadIdx.x] = k < 3 ? make_float2(P[OFF_W0 + 6 * i + k], P[OFF_W0 + 6 * i + 3 + k])
                                 : make_float2(P[OFF_B0 + 2 * i], P[OFF_B0 + 2 * i + 1]);
    }
    if (first) {
        mbar_init(mbar);
        *flag = 0;
    }
    if (threadIdx.x < 32) tc_alloc(slot, 128 * NWG);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tcols = *slot + (uint32_t)(g * WID);                         // this warpgroup's columns
    const uint32_t tl = tcols + ((uint32_t)(((threadIdx.x >> 5) & 3) * 32) << 16);  // + this warp's lanes
    const float4 *P4 = reinterpret_cast<const float4 *>(P);
    uint32_t parity = 0;
    bool ok = true;
    for (long long tile = (long long)g * gridDim.x + blockIdx.x; ok && tile * WID < n; tile += (long long)gridDim.x * NWG) {
        const long long row = tile * WID + tt;
        const bool valid = row < n;
        const float x0 = valid ? X[3 * row] : 0.f, x1 = valid ? X[3 * row + 1] : 0.f,
                    x2 = valid ? X[3 * row + 2] : 0.f;
        // input layer 3 -> 128 (FP32)
        const F2 xx0(x0), xx1(x1), xx2(x2);
#pragma unroll 2
        for (int c = part * (16 / PARTS); c < (part + 1) * (16 / PARTS); ++c) {
            F2 h[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(sin + 4 * (4 * c + i));
                const ulonglong2 wa = q[0], wb = q[1];
                F2 w0, w1, w2, bb;
                w0.v = wa.x; w1.v = wa.y; w2.v = wb.x; bb.v = wb.y;
                h[i] = gelu2(fma2(w0, xx0, fma2(w1, xx1, fma2(w2, xx2, bb))));
            }
            put8(sA, tt, 8 * c, h);
        }
        float y = 0.f;
        for (int l = 1; l <= 3; ++l) {
            ok = wg_gemm(sA, sB + (l - 1) * TILE_BYTES, tcols, mbar, parity, g, first, flag, err);
            if (!ok) break;
#pragma unroll 2
            for (int c = part * (8 / PARTS); c < (part + 1) * (8 / PARTS); ++c) {
                float v[16];
                tc_ld16(tl + (uint32_t)(c * 16), v);
                F2 h[8];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float4 q = __ldg(P4 + off_b(l) / 4 + 4 * c + k);
                    h[2 * k] = gelu2(add2(F2(v[4 * k], v[4 * k + 1]), F2(q.x, q.y)));
                    h[2 * k + 1] = gelu2(add2(F2(v[4 * k + 2], v[4 * k + 3]), F2(q.z, q.w)));
                }
                if (l < 3) {
                    put8(sA, tt, 16 * c, h);
                    put8(sA, tt, 16 * c + 8, h + 4);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 q = __ldg(P4 + OFF_W4 / 4 + 4 * c + k);
                        float a0, a1, a2, a3;
                        h[2 * k].get(a0, a1);
                        h[2 * k + 1].get(a2, a3);
                        y = fmaf(a0, q.x, y);
                        y = fmaf(a1, q.y, y);
                        y = fmaf(a2, q.z, y);
                        y = fmaf(a3, q.w, y);
                    }
                }
            }
        }
        // the second half's sum passes through the row's first chunk of the
        // activation tile, which only the first half's thread writes
        float *other = reinterpret_cast<float *>(sA + core_off(tt, 0));
        if (part == 1) *other = y;
        wg_bar(g);
        if (part == 0) y += *other;
        if (valid && ok && part == 0) Y[row] = y + P[OFF_B4];
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tc_dealloc(*slot, 128 * NWG);
}

// ------------------------------------------------------------- training
// One CTA of 16 warps per tile of ROWS batch rows: forward, backward, the
// tile's share of each gradient into its row of Gp [ntile][GSTRIDE] and its
// squared-error sum into Lp[tile]; k_mlp_reduce adds the tiles in a fixed
// order.  The output gradient dy = 2 (y - t) / B needs no sum across tiles, so
// the tiles are independent.
//
// The step is a chain of small layers, so its latency is the bound, not a
// rate: a tile is 16 or 32 rows (not the 128 an MMA would take as M), which
// spreads a batch of 256 over 16 CTAs, and every layer is computed
// transposed.  Features are the M dimension (TMEM lanes), batch rows the N
// dimension (columns), so all 16 warps share the element-wise work of a
// layer: thread (warp w, lane) owns feature o = 32 (w & 3) + lane of rows
// RPT (w >> 2) .. + RPT - 1, and its pre-activations of all layers stay in
// registers.  What a 128-row CTA of four warps took 345 us for (its
// pre-activations in global memory, each thread striding over its row, and
// operands transposed through 2-byte stores) takes 23 us for a batch of 256
// and 28 us for 4,096 (cold caches).
//
// One physical form of an operand serves every GEMM that reads it, as K-major
// or, transposed, as MN-major (instruction descriptor bits 15 and 16):
//   forward  z^T  = W a^T    A = W   (M = out, K = in)  B = a  (N = row, K = in)
//   input    dh^T = W^T dz^T A = W^T (M = in,  K = out) B = dz (N = row, K = out)
//   weights  gW   = dz^T a   A = dz^T (M = out, K = row) B = a^T (N = in, K = row)
// Tiles hold 8-row x 16-byte core matrices without swizzle: row group g and
// 16-byte chunk c at TG g + TC c, with the chunks 144 bytes apart so that the
// 2-byte stores of a warp (32 features of one row) fall on different banks.
// K-major: leading offset TC (next chunk along K), stride offset TG (next 8
// rows); MN-major: stride offset TC (next 8 along M or N), leading offset TG
// (next 8 along K).
constexpr uint32_t TC = 144, TG = 16 * TC;
constexpr uint32_t W_BYTES = 16 * TG;                      // 128 rows
constexpr uint32_t ID_BASE = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(WID >> 4) << 24);
__host__ __device__ constexpr uint32_t idesc_n(int n, int ta, int tb)
{
    return ID_BASE | ((uint32_t)ta << 15) | ((uint32_t)tb << 16) | ((uint32_t)(n >> 3) << 17);
}

__device__ __forceinline__ uint64_t desc_of(uint32_t saddr, uint32_t lead, uint32_t stride)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(lead >> 4) << 16) | ((uint64_t)(stride >> 4) << 32) |
           ((uint64_t)1 << 46);
}

__device__ __forceinline__ void mma_any(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, int accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

template <int N>
__device__ __forceinline__ void tc_ld_cols(uint32_t taddr, float *v)
{
    uint32_t r[N];
    if constexpr (N == 4) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(taddr));
    } else if constexpr (N == 16) {
        tc_ld16(taddr, v);
        return;
    } else {
        static_assert(N == 8, "4, 8 or 16 columns");
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                     : "r"(taddr));
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void cp_async16(uint32_t saddr, const void *g)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(saddr), "l"(g) : "memory");
}

constexpr int GRAD_THREADS = 512;
template <int ROWS> struct GradSmem {
    static constexpr uint32_t A_BYTES = (ROWS / 8) * TG;   // one activation tile
    static constexpr uint32_t OFF_A = 3 * W_BYTES;         // a0, a1, a2 (inputs of the hidden layers)
    static constexpr uint32_t OFF_DZ = OFF_A + 3 * A_BYTES;
    static constexpr uint32_t OFF_H = OFF_DZ + A_BYTES;    // FP32 [128][ROWS + 1]: last hidden layer
    static constexpr uint32_t OFF_SUM = OFF_H + 128 * (ROWS + 1) * 4;   // FP32 [4][128][4]: partial sums
    static constexpr uint32_t OFF_X = OFF_SUM + 4 * 128 * 4 * 4;        // FP32 [ROWS][4]: inputs, dy
    static constexpr uint32_t OFF_BAR = OFF_X + ROWS * 16; // 7 mbarriers, TMEM slot, flag
    static constexpr uint32_t BYTES = OFF_BAR + 128;
};

template <int ROWS>
__global__ void __launch_bounds__(GRAD_THREADS, 1) k_mlp_grad(Net net, const float *__restrict__ X,
                                                              const float *__restrict__ T, int B)
{
    using S = GradSmem<ROWS>;
    constexpr int RPT = ROWS / 4;             // rows of a thread
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    float *hbuf = reinterpret_cast<float *>(smem + S::OFF_H);
    float *sums = reinterpret_cast<float *>(smem + S::OFF_SUM);
    float4 *xs = reinterpret_cast<float4 *>(smem + S::OFF_X);
    uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + S::OFF_BAR);
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + S::OFF_BAR + 64);
    volatile int *flag = reinterpret_cast<int *>(smem + S::OFF_BAR + 72);
    const int t = threadIdx.x, w = t >> 5, cg = w >> 2;
    const int o = (w & 3) * 32 + (t & 31);    // this thread's feature
    const int r0 = blockIdx.x * ROWS;         // first batch row of the tile
    const float *__restrict__ P = net.P;
    float *__restrict__ Gp = net.Gp + (size_t)blockIdx.x * GSTRIDE;
    // the weight tiles, one copy group per layer
    for (int l = 0; l < 3; ++l) {
        for (int q = t; q < WID * 16; q += GRAD_THREADS) {
            const int r = q >> 4, c = q & 15;
            cp_async16(sbase + l * W_BYTES + (r >> 3) * TG + c * TC + (r & 7) * 16,
                       net.Wb + (l * WID + r) * WID + 8 * c);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    if (t < 7) mbar_init(mbar + t);
    if (t == 0) *flag = 0;
    if (w == 0) tc_alloc(slot, 512);
    if (t < ROWS) {
        const int row = r0 + t;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < B) { x.x = X[3 * row]; x.y = X[3 * row + 1]; x.z = X[3 * row + 2]; }
        xs[t] = x;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = *slot;
    const uint32_t lanes = (uint32_t)((w & 3) * 32) << 16;
    // TMEM: z_l / dh columns [0, 32), [32, 64), [64, 96); gW_l at 128 l (l = 1..3)
    const uint32_t zcol[3] = { tm, tm + 32u, tm + 64u };
    // one bf16 per row of this thread into a tile [row][feature]
    auto put = [&](uint32_t off, const float *v) {
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = cg * RPT + i;
            *reinterpret_cast<__nv_bfloat16 *>(smem + off + (r >> 3) * TG + (o >> 3) * TC + (r & 7) * 16 + (o & 7) * 2) =
                __float2bfloat16_rn(v[i]);
        }
    };
    // every thread waits for MMA group k; a timeout in any thread is seen by
    // all at the next barrier
    auto wait = [&](int k) {
        if (!mbar_wait(mbar + k, 0)) {
            *flag = 1;
            atomicOr(net.err, ERR_MMA_TIMEOUT);
            (void)mbar_wait(mbar + k, 0);
        }
        tc_fence_after();
    };
    float z[4][RPT];
    // ---------------- forward, the pre-activations kept
    {
        const float w0 = P[OFF_W0 + 3 * o], w1 = P[OFF_W0 + 3 * o + 1], w2 = P[OFF_W0 + 3 * o + 2], b0 = P[OFF_B0 + o];
        float h[RPT];
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const float4 x = xs[cg * RPT + i];
            z[0][i] = w0 * x.x + w1 * x.y + w2 * x.z + b0;
            h[i] = gelu(z[0][i]);
        }
        put(S::OFF_A, h);
    }
#pragma unroll
    for (int l = 1; l <= 3; ++l) {
        if (l == 1) asm volatile("cp.async.wait_group 2;\n" ::: "memory");
        else if (l == 2) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        proxy_fence();
        __syncthreads();
        if (t == 0) {
            tc_fence_after();
            const uint32_t a0 = sbase + (l - 1) * W_BYTES, b0 = sbase + S::OFF_A + (l - 1) * S::A_BYTES;
#pragma unroll
            for (int s = 0; s < 8; ++s)
                mma_any(zcol[l - 1], desc_of(a0 + s * 2 * TC, TC, TG), desc_of(b0 + s * 2 * TC, TC, TG),
                        idesc_n(ROWS, 0, 0), s > 0);
            mma_commit(mbar + l - 1);
        }
        const float bias = P[off_b(l) + o];
        wait(l - 1);
        float v[RPT], h[RPT];
        tc_ld_cols<RPT>(zcol[l - 1] + lanes + (uint32_t)(cg * RPT), v);
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            z[l][i] = v[i] + bias;
            h[i] = gelu(z[l][i]);
        }
        if (l < 3) {
            put(S::OFF_A + l * S::A_BYTES, h);
        } else {
#pragma unroll
            for (int i = 0; i < RPT; ++i) hbuf[o * (ROWS + 1) + cg * RPT + i] = h[i];
        }
        tc_fence_before();
    }
    __syncthreads();
    // output layer: the row's sum over the features in order, one thread per row
    if (w == 0) {
        float y = 0.f, dy = 0.f, sq = 0.f;
        const int row = r0 + t;
        if (t < ROWS && row < B) {
#pragma unroll 8
            for (int k = 0; k < WID; ++k) y += hbuf[k * (ROWS + 1) + t] * P[OFF_W4 + k];
            y += P[OFF_B4];
            dy = 2.0f * (y - T[row]) / (float)B;
            sq = (y - T[row]) * (y - T[row]);
        }
        if (t < ROWS) xs[t].w = dy;   // 0 on the rows past B
        float gb = dy;
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) {
            sq += __shfl_xor_sync(0xffffffffu, sq, k);
            gb += __shfl_xor_sync(0xffffffffu, gb, k);
        }
        if (t == 0) {
            net.Lp[blockIdx.x] = sq;
            Gp[OFF_B4] = gb;
        }
    }
    __syncthreads();
    // sums over a thread's rows of up to 4 values, then over the 4 row groups
    // in order: this thread's value `q` of feature o lands in sums[..]
    auto store_sum = [&](float4 v) { reinterpret_cast<float4 *>(sums)[cg * 128 + o] = v; };
    auto load_sum = [&]() {
        const float4 *q = reinterpret_cast<const float4 *>(sums);
        const float4 a = q[o], b = q[128 + o], c = q[256 + o], d = q[384 + o];
        return make_float4(((a.x + b.x) + c.x) + d.x, ((a.y + b.y) + c.y) + d.y, ((a.z + b.z) + c.z) + d.z,
                           ((a.w + b.w) + c.w) + d.w);
    };
    float dz[RPT];
    {
        const float w4 = P[OFF_W4 + o];
        float gw = 0.f, gb = 0.f;
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const float dy = xs[cg * RPT + i].w;
            dz[i] = dy * w4 * gelu_prime(z[3][i]);
            gw += dy * gelu(z[3][i]);
            gb += dz[i];
        }
        store_sum(make_float4(gw, gb, 0.f, 0.f));
    }
    // ---------------- hidden layers l = 3, 2, 1 (z_l = W_l a_{l-1} + b_l)
#pragma unroll
    for (int l = 3; l >= 1; --l) {
        put(S::OFF_DZ, dz);
        proxy_fence();
        tc_fence_before();
        __syncthreads();
        if (t == 0) {
            tc_fence_after();
            // input gradient first: the chain waits for it
            const uint32_t a0 = sbase + (l - 1) * W_BYTES, d0 = sbase + S::OFF_DZ;
#pragma unroll
            for (int s = 0; s < 8; ++s)
                mma_any(zcol[l - 1], desc_of(a0 + s * 2 * TG, TG, TC), desc_of(d0 + s * 2 * TC, TC, TG),
                        idesc_n(ROWS, 1, 0), s > 0);
            mma_commit(mbar + 6 - l);
            // the weight gradient: read from tensor memory at the end
            const uint32_t p0 = sbase + S::OFF_A + (l - 1) * S::A_BYTES;
#pragma unroll
            for (int s = 0; s < ROWS / 16; ++s)
                mma_any(tm + 128u * (uint32_t)l, desc_of(d0 + s * 2 * TG, TG, TC), desc_of(p0 + s * 2 * TG, TG, TC),
                        idesc_n(WID, 1, 1), s > 0);
            mma_commit(mbar + 6);
        }
        if (cg == 0) {
            const float4 v = load_sum();
            if (l == 3) {
                Gp[OFF_W4 + o] = v.x;
                Gp[off_b(3) + o] = v.y;
            } else {
                Gp[off_b(l) + o] = v.x;
            }
        }
        wait(6 - l);
        float v[RPT];
        tc_ld_cols<RPT>(zcol[l - 1] + lanes + (uint32_t)(cg * RPT), v);
        float g0 = 0.f, g1 = 0.f, g2 = 0.f, gb = 0.f;
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            dz[i] = v[i] * gelu_prime(z[l - 1][i]);
            gb += dz[i];
            if (l == 1) {
                const float4 x = xs[cg * RPT + i];
                g0 += dz[i] * x.x;
                g1 += dz[i] * x.y;
                g2 += dz[i] * x.z;
            }
        }
        // the weight-gradient MMAs still read the dz tile: wait for them before
        // the next layer's dz overwrites it
        if (!mbar_wait(mbar + 6, (uint32_t)(3 - l) & 1u)) {
            *flag = 1;
            atomicOr(net.err, ERR_MMA_TIMEOUT);
            (void)mbar_wait(mbar + 6, (uint32_t)(3 - l) & 1u);
        }
        __syncthreads();   // the sums above have been read
        store_sum(l == 1 ? make_float4(gb, g0, g1, g2) : make_float4(gb, 0.f, 0.f, 0.f));
    }
    tc_fence_after();
    __syncthreads();
    if (cg == 0) {
        // input layer
        const float4 v = load_sum();
        Gp[OFF_B0 + o] = v.x;
        Gp[OFF_W0 + 3 * o] = v.y;
        Gp[OFF_W0 + 3 * o + 1] = v.z;
        Gp[OFF_W0 + 3 * o + 2] = v.w;
    }
    if (*flag == 0) {
        // the weight gradients: lane = output unit, columns = inputs
#pragma unroll
        for (int l = 1; l <= 3; ++l) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float v[8];
                tc_ld_cols<8>(tm + 128u * (uint32_t)l + lanes + (uint32_t)(cg * 32 + c * 8), v);
                float4 *dst = reinterpret_cast<float4 *>(Gp + off_W(l) + o * WID + cg * 32 + c * 8);
                dst[0] = make_float4(v[0], v[1], v[2], v[3]);
                dst[1] = make_float4(v[4], v[5], v[6], v[7]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (w == 0) tc_dealloc(tm, 512);
}

// Inference of few rows: a tile of ROWS (16, 32 or 64) rows per CTA in the
// gradient kernel's transposed form, so the chain of layers is short and the
// 16 warps of every SM take part.  Bound by latency: the weights' way into
// shared memory and four layers in turn.  Calls back to back: 1,001 rows take
// 10.3 us (18.5 us in 128-row tiles), 5,000 rows 13.2 us (20.0 us).  Same
// operations per row as above, in the same order.
template <int ROWS> struct RowsSmem {
    static constexpr uint32_t A_BYTES = (ROWS / 8) * TG;
    static constexpr uint32_t OFF_A = 3 * W_BYTES;         // two activation tiles, in turn
    static constexpr uint32_t OFF_H = OFF_A + 2 * A_BYTES; // FP32 [128][ROWS + 1]: last hidden layer
    static constexpr uint32_t OFF_X = OFF_H + 128 * (ROWS + 1) * 4;
    static constexpr uint32_t OFF_BAR = OFF_X + ROWS * 16; // 3 mbarriers, TMEM slot, flag
    static constexpr uint32_t BYTES = OFF_BAR + 128;
};

template <int ROWS>
__global__ void __launch_bounds__(GRAD_THREADS, 1) k_mlp_rows(const float *__restrict__ P,
                                                              const __nv_bfloat16 *__restrict__ Wb,
                                                              const float *__restrict__ X, float *__restrict__ Y,
                                                              long long n, int *err)
{
    using S = RowsSmem<ROWS>;
    constexpr int RPT = ROWS / 4;             // rows of a thread
    extern __shared__ __align__(1024) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    float *hbuf = reinterpret_cast<float *>(smem + S::OFF_H);
    float4 *xs = reinterpret_cast<float4 *>(smem + S::OFF_X);
    uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + S::OFF_BAR);
    uint32_t *slot = reinterpret_cast<uint32_t *>(smem + S::OFF_BAR + 64);
    volatile int *flag = reinterpret_cast<int *>(smem + S::OFF_BAR + 72);
    const int t = threadIdx.x, w = t >> 5, cg = w >> 2;
    const int o = (w & 3) * 32 + (t & 31);    // this thread's feature
    const long long r0 = (long long)blockIdx.x * ROWS;
    // the weight tiles, one copy group per layer
    for (int l = 0; l < 3; ++l) {
        for (int q = t; q < WID * 16; q += GRAD_THREADS) {
            const int r = q >> 4, c = q & 15;
            cp_async16(sbase + l * W_BYTES + (r >> 3) * TG + c * TC + (r & 7) * 16, Wb + (l * WID + r) * WID + 8 * c);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    if (t < 3) mbar_init(mbar + t);
    if (t == 0) *flag = 0;
    if (w == 0) tc_alloc(slot, 64);
    if (t < ROWS) {
        const long long row = r0 + t;
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < n) { x.x = X[3 * row]; x.y = X[3 * row + 1]; x.z = X[3 * row + 2]; }
        xs[t] = x;
    }
    const float w0 = P[OFF_W0 + 3 * o], w1 = P[OFF_W0 + 3 * o + 1], w2 = P[OFF_W0 + 3 * o + 2];
    const float b[4] = { P[OFF_B0 + o], P[off_b(1) + o], P[off_b(2) + o], P[off_b(3) + o] };
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tm = *slot;
    const uint32_t lanes = (uint32_t)((w & 3) * 32) << 16;
    // this thread's feature of its rows, two at a time, into a tile [row][feature]
    auto put = [&](uint32_t off, const F2 *v) {
#pragma unroll
        for (int i = 0; i < RPT; i += 2) {
            const int r = cg * RPT + i;
            float a0, a1;
            v[i / 2].get(a0, a1);
            __nv_bfloat16 *q = reinterpret_cast<__nv_bfloat16 *>(smem + off + (r >> 3) * TG + (o >> 3) * TC + (r & 7) * 16 +
                                                                 (o & 7) * 2);
            q[0] = __float2bfloat16_rn(a0);
            q[8] = __float2bfloat16_rn(a1);   // the next row: 16 bytes on
        }
    };
    {
        F2 h[RPT / 2];
#pragma unroll
        for (int i = 0; i < RPT / 2; ++i) {
            const float4 p = xs[cg * RPT + 2 * i], q = xs[cg * RPT + 2 * i + 1];
            h[i] = gelu2(fma2(F2(w0), F2(p.x, q.x), fma2(F2(w1), F2(p.y, q.y), fma2(F2(w2), F2(p.z, q.z), F2(b[0])))));
        }
        put(S::OFF_A, h);
    }
#pragma unroll
    for (int l = 1; l <= 3; ++l) {
        if (l == 1) asm volatile("cp.async.wait_group 2;\n" ::: "memory");
        else if (l == 2) asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        else asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        proxy_fence();
        __syncthreads();
        if (t == 0) {
            tc_fence_after();
            const uint32_t a0 = sbase + (l - 1) * W_BYTES, b0 = sbase + S::OFF_A + ((l - 1) & 1) * S::A_BYTES;
#pragma unroll
            for (int s = 0; s < 8; ++s)
                mma_any(tm, desc_of(a0 + s * 2 * TC, TC, TG), desc_of(b0 + s * 2 * TC, TC, TG), idesc_n(ROWS, 0, 0), s > 0);
            mma_commit(mbar + l - 1);
        }
        if (!mbar_wait(mbar + l - 1, 0)) {
            *flag = 1;
            atomicOr(err, ERR_MMA_TIMEOUT);
            (void)mbar_wait(mbar + l - 1, 0);
        }
        tc_fence_after();
        float v[RPT];
        F2 h[RPT / 2];
        tc_ld_cols<RPT>(tm + lanes + (uint32_t)(cg * RPT), v);
#pragma unroll
        for (int i = 0; i < RPT / 2; ++i) h[i] = gelu2(add2(F2(v[2 * i], v[2 * i + 1]), F2(b[l])));
        if (l < 3) {
            put(S::OFF_A + (l & 1) * S::A_BYTES, h);
        } else {
#pragma unroll
            for (int i = 0; i < RPT / 2; ++i) {
                float a0, a1;
                h[i].get(a0, a1);
                hbuf[o * (ROWS + 1) + cg * RPT + 2 * i] = a0;
                hbuf[o * (ROWS + 1) + cg * RPT + 2 * i + 1] = a1;
            }
        }
        tc_fence_before();
    }
    __syncthreads();
    // output layer: the row's sum over the features in order, one thread per row
    if (t < ROWS && r0 + t < n && *flag == 0) {
        float y = 0.f, y1 = 0.f;
#pragma unroll 16
        for (int k = 0; k < WID / 2; ++k) {
            y = fmaf(hbuf[k * (ROWS + 1) + t], __ldg(P + OFF_W4 + k), y);
            y1 = fmaf(hbuf[(k + WID / 2) * (ROWS + 1) + t], __ldg(P + OFF_W4 + WID / 2 + k), y1);
        }
        Y[r0 + t] = (y + y1) + P[OFF_B4];
    }
    if (w == 0) tc_dealloc(tm, 64);
}

// Gradient and loss of the batch: the tiles' shares added in tile order.  The
// loads of SHARES tiles stand before their additions, and the loss is a
// thread's of its own: a chain of loads eight at a time, twice on the thread
// that also had the loss, was part of the 14.3 us of 128 tiles (11.5 us now,
// cold; 16 tiles with Adam 4.7 us).
__device__ __forceinline__ float tile_sum(const float *__restrict__ q, size_t stride, int ntile)
{
    constexpr int SHARES = 32;
    float g = 0.f;
    for (int i0 = 0; i0 < ntile; i0 += SHARES) {
        float v[SHARES];
#pragma unroll
        for (int i = 0; i < SHARES; ++i) v[i] = i0 + i < ntile ? q[(size_t)(i0 + i) * stride] : 0.f;
#pragma unroll
        for (int i = 0; i < SHARES; ++i) g += v[i];
    }
    return g;
}
__device__ __forceinline__ void loss_of(const Net &net, int ntile, int B) { *net.loss = tile_sum(net.Lp, 1, ntile) / (float)B; }

__global__ void k_mlp_reduce(Net net, int ntile, int B)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < NPARAM) net.G[k] = tile_sum(net.Gp + k, GSTRIDE, ntile);
    else if (k == NPARAM) loss_of(net, ntile, B);
}

// The same sums followed by Adam (Kingma & Ba) on the FP32 masters; refreshes
// the BF16 copies.
__global__ void k_mlp_reduce_adam(Net net, int ntile, int B, float lr, float b1, float b2, float eps, float c1, float c2)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k == NPARAM) loss_of(net, ntile, B);
    if (k >= NPARAM) return;
    const float m0 = net.M[k], v0 = net.V[k], p0 = net.P[k];
    const float g = tile_sum(net.Gp + k, GSTRIDE, ntile);
    net.G[k] = g;
    const float m = b1 * m0 + (1.f - b1) * g;
    const float v = b2 * v0 + (1.f - b2) * g * g;
    net.M[k] = m;
    net.V[k] = v;
    const float p = p0 - lr * (m / c1) / (sqrtf(v / c2) + eps);
    net.P[k] = p;
    for (int l = 1; l <= 3; ++l)
        if (k >= off_W(l) && k < off_W(l) + WID * WID) net.Wb[(l - 1) * WID * WID + (k - off_W(l))] = __float2bfloat16_rn(p);
}

__global__ void k_mlp_refresh(Net net)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 3 * WID * WID) return;
    const int l = k / (WID * WID) + 1, e = k % (WID * WID);
    net.Wb[k] = __float2bfloat16_rn(net.P[off_W(l) + e]);
}

}  // namespace mlp
}  // namespace sdpd

// ======================================================================= ABI
using namespace sdpd::mlp;

struct sdpd_mlp {
    Net net;
};

namespace {
// Batch rows per CTA of the gradient kernel: 16 up to 512 rows (more CTAs and
// a shorter chain each), 32 beyond (half the gradient shares to add).
constexpr int SMALL_ROWS = 512;
int grad_tiles(int batch) { return batch <= SMALL_ROWS ? (batch + 15) / 16 : (batch + 31) / 32; }
int grad_tiles_max(int bmax) { return std::max(grad_tiles(std::min(bmax, SMALL_ROWS)), grad_tiles(bmax)); }

sdpd_status mlp_fail(sdpd_status s, const std::string &m)
{
    sdpd::set_last_error(m.c_str());
    return s;
}

sdpd_status mlp_err(sdpd_mlp *h)
{
    int e = 0;
    if (cudaMemcpy(&e, h->net.err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
        return mlp_fail(SDPD_E_CUDA, "mlp: reading the error word");
    if (e) return mlp_fail(SDPD_E_TIMEOUT, "mlp: tensor-core completion wait timed out");
    return SDPD_OK;
}
sdpd_status launch_grad(sdpd_mlp *h, const float *X, const float *T, int batch, cudaStream_t st)
{
    (void)cudaGetLastError();
    const int ntile = grad_tiles(batch);
    if (batch <= SMALL_ROWS)
        k_mlp_grad<16><<<ntile, GRAD_THREADS, GradSmem<16>::BYTES, st>>>(h->net, X, T, batch);
    else
        k_mlp_grad<32><<<ntile, GRAD_THREADS, GradSmem<32>::BYTES, st>>>(h->net, X, T, batch);
    return cudaGetLastError() == cudaSuccess ? SDPD_OK : mlp_fail(SDPD_E_CUDA, "mlp_gradients: launch");
}

sdpd_status read_loss(sdpd_mlp *h, float *loss, cudaStream_t st, const char *what)
{
    if (cudaMemcpyAsync(loss, h->net.loss, 4, cudaMemcpyDefault, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return mlp_fail(SDPD_E_CUDA, what);
    return mlp_err(h);
}
}  // namespace

extern "C" {

void mlp_destroy(sdpd_mlp *h);

sdpd_status mlp_init(int in, int width, int depth, unsigned long long seed, int batch_max, sdpd_mlp **out)
{
    if (!out) return mlp_fail(SDPD_E_INVALID, "mlp_init: out is NULL");
    *out = nullptr;
    if (in != NIN || width != WID || depth != 4) return mlp_fail(SDPD_E_INVALID, "mlp_init: network is 3 -> 4 x 128 -> 1");
    if (batch_max < 1 || batch_max > 4096) return mlp_fail(SDPD_E_INVALID, "mlp_init: batch_max must be 1..4096");
    sdpd_mlp *h = new sdpd_mlp();
    Net &n = h->net;
    n.bmax = (batch_max + WID - 1) / WID * WID;
    auto A = [&](void **p, size_t bytes) { return cudaMalloc(p, bytes) == cudaSuccess; };
    bool ok = A((void **)&n.P, NPARAM * 4) && A((void **)&n.G, NPARAM * 4) && A((void **)&n.M, NPARAM * 4) &&
              A((void **)&n.V, NPARAM * 4) && A((void **)&n.Wb, 3 * WID * WID * 2) &&
              A((void **)&n.Gp, (size_t)grad_tiles_max(n.bmax) * GSTRIDE * 4) &&
              A((void **)&n.Lp, (size_t)grad_tiles_max(n.bmax) * 4) && A((void **)&n.loss, 4) && A((void **)&n.err, 4);
    if (!ok) {
        delete h;
        return mlp_fail(SDPD_E_OOM, "mlp_init: cudaMalloc failed");
    }
    // He-uniform initial weights from a splitmix64 stream of the seed
    std::vector<float> P(NPARAM, 0.f);
    uint64_t st = seed ^ 0x9E3779B97F4A7C15ull;
    auto rnd = [&]() {
        st += 0x9E3779B97F4A7C15ull;
        uint64_t z = st;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return (double)(z >> 11) * (1.0 / 9007199254740992.0);
    };
    auto fill = [&](int off, int count, int fan_in) {
        const double lim = std::sqrt(6.0 / fan_in);
        for (int k = 0; k < count; ++k) P[off + k] = (float)((2.0 * rnd() - 1.0) * lim);
    };
    fill(OFF_W0, WID * NIN, NIN);
    for (int l = 1; l <= 3; ++l) fill(off_W(l), WID * WID, WID);
    fill(OFF_W4, WID, WID);
    cudaMemcpy(n.P, P.data(), NPARAM * 4, cudaMemcpyHostToDevice);
    cudaMemset(n.M, 0, NPARAM * 4);
    cudaMemset(n.V, 0, NPARAM * 4);
    cudaMemset(n.G, 0, NPARAM * 4);
    cudaMemset(n.err, 0, 4);
    n.step = 0;
    k_mlp_refresh<<<(3 * WID * WID + 255) / 256, 256>>>(n);
    cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FWD_SMEM);
    cudaFuncSetAttribute(k_mlp_rows<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RowsSmem<16>::BYTES);
    cudaFuncSetAttribute(k_mlp_rows<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RowsSmem<32>::BYTES);
    cudaFuncSetAttribute(k_mlp_rows<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RowsSmem<64>::BYTES);
    cudaFuncSetAttribute(k_mlp_grad<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GradSmem<16>::BYTES);
    cudaFuncSetAttribute(k_mlp_grad<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GradSmem<32>::BYTES);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        mlp_destroy(h);
        return mlp_fail(SDPD_E_CUDA, "mlp_init: initialisation failed");
    }
    *out = h;
    return SDPD_OK;
}

void mlp_destroy(sdpd_mlp *h)
{
    if (!h) return;
    cudaDeviceSynchronize();
    Net &n = h->net;
    void *ps[] = { n.P, n.G, n.M, n.V, n.Wb, n.Gp, n.Lp, n.loss, n.err };
    for (void *p : ps) cudaFree(p);
    delete h;
}

sdpd_status mlp_set_params(sdpd_mlp *h, const float *params)
{
    if (!h || !params) return mlp_fail(SDPD_E_INVALID, "mlp_set_params: NULL argument");
    if (cudaMemcpy(h->net.P, params, NPARAM * 4, cudaMemcpyDefault) != cudaSuccess)
        return mlp_fail(SDPD_E_CUDA, "mlp_set_params: copy");
    k_mlp_refresh<<<(3 * WID * WID + 255) / 256, 256>>>(h->net);
    cudaMemset(h->net.M, 0, NPARAM * 4);
    cudaMemset(h->net.V, 0, NPARAM * 4);
    h->net.step = 0;
    return cudaDeviceSynchronize() == cudaSuccess ? SDPD_OK : mlp_fail(SDPD_E_CUDA, "mlp_set_params");
}

sdpd_status mlp_get_params(sdpd_mlp *h, float *params, float *grads)
{
    if (!h) return mlp_fail(SDPD_E_INVALID, "mlp_get_params: NULL argument");
    if (cudaDeviceSynchronize() != cudaSuccess) return mlp_fail(SDPD_E_CUDA, "mlp_get_params");
    if (params && cudaMemcpy(params, h->net.P, NPARAM * 4, cudaMemcpyDefault) != cudaSuccess)
        return mlp_fail(SDPD_E_CUDA, "mlp_get_params: copy");
    if (grads && cudaMemcpy(grads, h->net.G, NPARAM * 4, cudaMemcpyDefault) != cudaSuccess)
        return mlp_fail(SDPD_E_CUDA, "mlp_get_params: copy");
    return SDPD_OK;
}

int mlp_param_count(void) { return NPARAM; }

sdpd_status mlp_gradients(sdpd_mlp *h, const float *X, const float *T, int batch, float *loss, void *stream)
{
    if (!h || !X || !T) return mlp_fail(SDPD_E_INVALID, "mlp_gradients: NULL argument");
    if (batch < 1 || batch > h->net.bmax) return mlp_fail(SDPD_E_INVALID, "mlp_gradients: batch out of range");
    cudaStream_t st = (cudaStream_t)stream;
    const sdpd_status s = launch_grad(h, X, T, batch, st);
    if (s != SDPD_OK) return s;
    k_mlp_reduce<<<(NPARAM + 255) / 256, 256, 0, st>>>(h->net, grad_tiles(batch), batch);
    if (cudaGetLastError() != cudaSuccess) return mlp_fail(SDPD_E_CUDA, "mlp_gradients: launch");
    return loss ? read_loss(h, loss, st, "mlp_gradients: loss") : SDPD_OK;
}

sdpd_status mlp_train_step(sdpd_mlp *h, const float *X, const float *T, int batch, float lr, float *loss,
                           void *stream)
{
    if (!h || !X || !T) return mlp_fail(SDPD_E_INVALID, "mlp_gradients: NULL argument");
    if (batch < 1 || batch > h->net.bmax) return mlp_fail(SDPD_E_INVALID, "mlp_gradients: batch out of range");
    cudaStream_t st = (cudaStream_t)stream;
    const sdpd_status s = launch_grad(h, X, T, batch, st);
    if (s != SDPD_OK) return s;
    h->net.step += 1;
    const double b1 = 0.9, b2 = 0.999;
    const float c1 = (float)(1.0 - std::pow(b1, (double)h->net.step));
    const float c2 = (float)(1.0 - std::pow(b2, (double)h->net.step));
    k_mlp_reduce_adam<<<(NPARAM + 255) / 256, 256, 0, st>>>(h->net, grad_tiles(batch), batch, lr, (float)b1, (float)b2,
                                                           1e-8f, c1, c2);
    if (cudaGetLastError() != cudaSuccess) return mlp_fail(SDPD_E_CUDA, "mlp_train_step: launch");
    return loss ? read_loss(h, loss, st, "mlp_train_step: loss") : SDPD_OK;
}

sdpd_status mlp_infer(sdpd_mlp *h, const float *X, float *Y, long long n, void *stream)
{
    if (!h || (n && (!X || !Y))) return mlp_fail(SDPD_E_INVALID, "mlp_infer: NULL argument");
    if (n <= 0) return SDPD_OK;
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaStream_t st = (cudaStream_t)stream;
    (void)cudaGetLastError();
    // The smallest tile that covers the rows with one CTA per SM: a call of a
    // given size takes the longer the larger its tiles (calls of 1,001 rows back
    // to back: 10.3 us in tiles of 16 or 32, 12.3 of 64, 18.5 of 128), and a second
    // round of small ones costs more than the next size up (2,500 rows: 18.4 of
    // 16, 12.3 of 32; 5,000: 18.5 of 32, 13.2 of 64; 10,000: 22.5 of 64, 20.5 of
    // 128).
    const int rows = n <= 16LL * nsm ? 16 : n <= 32LL * nsm ? 32 : n <= 64LL * nsm ? 64 : WID;
    const unsigned grid = (unsigned)std::min<long long>((n + rows - 1) / rows, nsm);
    const Net &N = h->net;
    if (rows == 16)
        k_mlp_rows<16><<<grid, GRAD_THREADS, RowsSmem<16>::BYTES, st>>>(N.P, N.Wb, X, Y, n, N.err);
    else if (rows == 32)
        k_mlp_rows<32><<<grid, GRAD_THREADS, RowsSmem<32>::BYTES, st>>>(N.P, N.Wb, X, Y, n, N.err);
    else if (rows == 64)
        k_mlp_rows<64><<<grid, GRAD_THREADS, RowsSmem<64>::BYTES, st>>>(N.P, N.Wb, X, Y, n, N.err);
    else
        k_mlp_forward<<<grid, FWD_GROUP * NWG, FWD_SMEM, st>>>(N.P, N.Wb, X, Y, n, N.err);
    if (cudaGetLastError() != cudaSuccess) return mlp_fail(SDPD_E_CUDA, "mlp_infer: launch");
    return SDPD_OK;
}

sdpd_status mlp_check(sdpd_mlp *h)
{
    if (!h) return mlp_fail(SDPD_E_INVALID, "mlp_check: NULL");
    if (cudaDeviceSynchronize() != cudaSuccess) return mlp_fail(SDPD_E_CUDA, "mlp_check: device error");
    return mlp_err(h);
}

}  // extern "C"
