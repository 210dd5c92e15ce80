// mlp.cu -- the learned swarm proposal's network on the 5th-generation tensor
// cores.  Not part of the paper (Sec. 6 names learned priors as future work): a
// 4-layer MLP 832 -> 256 -> 256 -> 256 -> 16 whose output seeds the PST of a
// frame (the c_0, r_0 of the Sec. 4 initialisation).  Training (forward, loss,
// backward, Adam) and inference run only the kernels of this file.
//
// Forward passes of up to 8 rows are one launch of forward_small_kernel.  Every other
// product is a part of a launch of umma_gemm_kernel:
//     C[M x N] = A[M x K] . B[N x K]^T,  A, B bfloat16 row-major (K contiguous),
//     FP32 accumulation in tensor memory (TMEM), fused epilogue.
// A forward layer is a launch of its own; a backward launch holds a layer's weight and
// input gradients and its bias gradient (the first one also the total of the loss).
// One CTA owns a 128 x 32 tile of C and 32 TMEM columns:
//   warp 0, lane 0   TMA producer: 64-column slabs of A (128 rows) and B (32 rows)
//                    into a 5-stage shared-memory ring (mbarrier transaction
//                    counts), one box of 128-byte rows per operand and slab
//   warp 1, lane 0   MMA issuer: 4 x tcgen05.mma.kind::f16 (M 128, N 32, K 16)
//                    per slab; tcgen05.commit releases the slab
//   warps 0..3       epilogue: tcgen05.ld of the warp's 32 accumulator lanes,
//                    bias / ReLU / gradient mask, bfloat16 or FP32 stores, the
//                    bfloat16 ones optionally also transposed (the backward
//                    products reduce over the batch and need batch-contiguous
//                    operands)
// The products are tiny (K <= 1024, at most 16 tiles of 128 x 128 at a training batch
// of 1024), so a launch is bound by its chain of loads, products and epilogue, not by
// tensor throughput.  Boxes of whole 128-byte rows move a slab in 2 TMA requests of
// 160 rows; with unswizzled boxes of 16-byte rows the 16 requests of 128 rows were the
// main loop's limit.  The narrow tile gives four times the CTAs of a 128 x 128 one and
// a quarter of its epilogue.  Measured, gradient of 512 rows / forward of 1 / 4096
// rows: 16-byte boxes, 128 x 128 tile 270 / 56 / 62 us; 128-byte boxes, tile N 128:
// 219 / 38 / 41, N 64: 170 / 30 / 35, N 32: 150 / 29 / 44, N 16: 135 / 27 / 68.  Five
// stages rather than eight leave room for two CTAs on an SM, so that the next launch of a
// chain can set up beside this one; with that and its operands of the epilogue fetched
// before the products are done, a forward pass takes 21 us at 9 rows and 26 at 4096.
// Shared-memory operand layout: K-major with the 128-byte swizzle that TMA writes and
// the MMA reads -- a slab row is 128 bytes, eight rows are one 1024-byte atom, so the
// stride-dimension (M/N) byte offset is 1024, the leading-dimension offset is unused,
// tiles are 1024-byte aligned, and K step j of a slab starts 32 j bytes in.  Every wait
// on an mbarrier is bounded in time; on expiry the CTA records RF_ERR_TIMEOUT, lets its
// copies land, frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "rf_proposal.h"

namespace rf {
namespace {

typedef __nv_bfloat16 bf16;

constexpr int GB_M = 128, GB_N = 32, GB_K = 64, GB_STAGES = 5, GB_THREADS = 128;
constexpr int GB_ROW = 2 * GB_K;            // bytes of a slab row: one swizzle row
constexpr int GB_TILE_A = GB_M * GB_ROW, GB_TILE_B = GB_N * GB_ROW;
constexpr int GB_STAGE = GB_TILE_A + GB_TILE_B;
constexpr int GB_SBO = 8 * GB_ROW;          // M/N-direction step: eight rows
constexpr int GB_BAR_OFF = GB_STAGES * GB_STAGE;
constexpr int GB_SMEM = GB_BAR_OFF + 256 + 1024;  // + barriers, + alignment slack
constexpr uint32_t GB_TMEM_COLS = 32;
static_assert(GB_TILE_A % 1024 == 0 && GB_TILE_B % 1024 == 0, "swizzle atoms");
// kind::f16 instruction descriptor: D FP32 (bits 4-5 = 1), A and B bfloat16
// (bits 7-9 = 1, 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
constexpr uint32_t GB_IDESC =
    (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(GB_N >> 3) << 17) | ((uint32_t)(GB_M >> 4) << 24);

enum { EPI_BIAS_RELU = 0, EPI_BIAS = 1, EPI_MASK = 2, EPI_PLAIN = 3, EPI_LOSS = 4 };

struct GemmEpi {
    int M, N, K;           // N a multiple of 16
    int mode;
    const float *bias;     // [N], 16-byte aligned (EPI_BIAS_RELU, EPI_BIAS, EPI_LOSS)
    const bf16 *mask;      // [M x N], ld_mask    (EPI_MASK: keep where mask > 0)
    bf16 *out_h;           // [M x N] bfloat16, ld_h (may be NULL)
    bf16 *out_ht;          // [N x M] bfloat16, ld_ht (may be NULL)
    float *out_f;          // [M x N] FP32, ld_f (may be NULL)
    int ld_mask, ld_h, ld_ht, ld_f;
    const bf16 *x;         // EPI_LOSS: the batch inputs and targets; out_h / out_ht receive
    const float *y;        //   the gradient of the outputs, out_f the outputs
    double *loss_part;     //   [ceil(M / 32)] loss sums of 32 rows
    int *err;
    long long timeout_ns;
};

// One launch: the CTAs of one or two products of the same inputs, then (backward)
// those of a bias gradient, then one that totals the loss.
struct GemmArgs {
    CUtensorMap ta[2], tb[2];
    GemmEpi e[2];
    int tiles[2];          // CTAs of each product
    const bf16 *bias_dt;   // [bias_n x bias_b] transposed gradient, its row sums to bias_db
    float *bias_db;
    int bias_n, bias_b;
    const double *loss_part;
    float *loss;           // mean loss of loss_rows rows (NULL: no such CTA)
    int loss_rows;
};

// ------------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ long long gtimer()
{
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}

// Wait for the phase of `parity` to complete; false after timeout_ns.
__device__ bool mbar_wait(uint32_t bar, uint32_t parity, long long timeout_ns)
{
    if (mbar_try_wait(bar, parity))
        return true;
    const long long t0 = gtimer();
    while (!mbar_try_wait(bar, parity))
        if (gtimer() - t0 > timeout_ns)
            return false;
    return true;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 ::"r"(dst), "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: start >> 4 (bits 0-13), leading byte offset
// >> 4 (16-29, unused with a swizzle), stride byte offset >> 4 (32-45), the fixed
// 0b001 of bits 46-48, base offset 0, swizzle mode 2 (128 bytes, bits 61-63).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(GB_SBO >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t acc)
{
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(GB_IDESC), "r"(acc)
                 : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 16 consecutive FP32 accumulator columns of this thread's TMEM lane; the wait
// sits in the same statement so the registers are valid when it returns.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16])
{
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15}, [%16];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i)
        v[i] = __uint_as_float(r[i]);
}

// K steps of 16 of slab kb that hold data (the rest of the slab is zero fill).
__device__ __forceinline__ int slab_steps(int K, int kb) { return (min(GB_K, K - kb * GB_K) + 15) >> 4; }

// ------------------------------------------------------------------ epilogue
__device__ __forceinline__ void store_bf16(const GemmEpi &e, int m, int n, const float v[16])
{
    bf16 h[16];
#pragma unroll
    for (int i = 0; i < 16; ++i)
        h[i] = __float2bfloat16_rn(v[i]);
    if (e.out_h) {
        uint4 q[2];
        memcpy(q, h, sizeof q);
        uint4 *o = reinterpret_cast<uint4 *>(e.out_h + (size_t)m * e.ld_h + n);
        o[0] = q[0];
        o[1] = q[1];
    }
    if (e.out_ht)  // lanes hold consecutive m: each column store is coalesced
#pragma unroll
        for (int i = 0; i < 16; ++i)
            e.out_ht[(size_t)(n + i) * e.ld_ht + m] = h[i];
}

// What the epilogue of row m, columns n0 .. n0 + GB_N reads, fetched while the products run.
struct EpiInputs {
    float bias[GB_N];
    uint4 q[GB_N / 8];     // EPI_MASK: the mask row; EPI_LOSS: q[0] the previous offset, then y
};

__device__ __forceinline__ void epi_fetch(const GemmEpi &e, int m, int n0, EpiInputs &in)
{
    const bool has_bias = e.mode == EPI_BIAS_RELU || e.mode == EPI_BIAS || e.mode == EPI_LOSS;
#pragma unroll
    for (int i = 0; i < GB_N; i += 4) {
        const float4 b = has_bias && n0 + i < e.N ? __ldg(reinterpret_cast<const float4 *>(e.bias + n0 + i))
                                                  : make_float4(0.f, 0.f, 0.f, 0.f);
        in.bias[i] = b.x;
        in.bias[i + 1] = b.y;
        in.bias[i + 2] = b.z;
        in.bias[i + 3] = b.w;
    }
#pragma unroll
    for (int i = 0; i < GB_N / 8; ++i)
        in.q[i] = make_uint4(0, 0, 0, 0);
    if (m >= e.M)
        return;
    if (e.mode == EPI_MASK) {
        const uint4 *mk = reinterpret_cast<const uint4 *>(e.mask + (size_t)m * e.ld_mask + n0);
#pragma unroll
        for (int i = 0; i < GB_N / 8; ++i)
            if (n0 + 8 * i < e.N)
                in.q[i] = mk[i];
    } else if (e.mode == EPI_LOSS) {
        in.q[0] = *reinterpret_cast<const uint4 *>(e.x + (size_t)m * RF_MLP_IN + RF_MLP_IN_USED - 6);
        const uint2 *y = reinterpret_cast<const uint2 *>(e.y + (size_t)m * 6);
        const uint2 a = y[0], b = y[1], c = y[2];
        in.q[1] = make_uint4(a.x, a.y, b.x, b.y);
        in.q[2] = make_uint4(c.x, c.y, 0, 0);
    }
}

// Loss (mean over the batch of sum_d 1/2 r^2 (1 + e^{-2s}) + s, r = y - mu,
// mu = x_v + o_mu with x_v the previous-offset inputs (columns 768..773 of the
// batch rows), s = clamp(o_s, -6, 6)) of one row and, in v, its gradient with
// respect to the 16 outputs in FP32.
__device__ __forceinline__ float loss_row(const EpiInputs &in, int B, float v[16])
{
    bf16 xv[8];
    float y[8];
    memcpy(xv, &in.q[0], sizeof xv);
    memcpy(y, &in.q[1], sizeof y);
    float gr[RF_MLP_OUT];
#pragma unroll
    for (int j = 0; j < RF_MLP_OUT; ++j)
        gr[j] = 0.f;
    const float inv_b = 1.f / (float)B;
    float lf = 0.f;
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        const float mu = v[d] + __bfloat162float(xv[d]);
        const float sr = v[6 + d];
        const float s = fminf(fmaxf(sr, -6.f), 6.f);
        const float r = y[d] - mu;
        const float ex = expf(-2.f * s);
        lf += 0.5f * r * r * (1.f + ex) + s;
        gr[d] = -r * (1.f + ex) * inv_b;
        gr[6 + d] = (sr > -6.f && sr < 6.f) ? (1.f - r * r * ex) * inv_b : 0.f;
    }
#pragma unroll
    for (int j = 0; j < RF_MLP_OUT; ++j)
        v[j] = gr[j];
    return lf;
}

// Columns n .. n + 16 of row m (n = n0 + nc); called by whole warps.
__device__ __forceinline__ void epi_store(const GemmEpi &e, int m, int n, int nc, const EpiInputs &in, float v[16])
{
    const bool live = m < e.M;
    if (e.mode == EPI_MASK) {
        bf16 mk[16];
        memcpy(mk, &in.q[nc / 8], sizeof mk);
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (!(__bfloat162float(mk[i]) > 0.f))
                v[i] = 0.f;
    } else if (e.mode != EPI_PLAIN) {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            v[i] += in.bias[nc + i];
            if (e.mode == EPI_BIAS_RELU)
                v[i] = fmaxf(v[i], 0.f);
        }
    }
    if (e.out_f && live) {
        float *o = e.out_f + (size_t)m * e.ld_f + n;
#pragma unroll
        for (int i = 0; i < 16; i += 4)
            *reinterpret_cast<float4 *>(o + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
    if (e.mode == EPI_LOSS) {  // row sums in FP64, in a fixed order: 32 rows here, then the warps'
        double l = live ? (double)loss_row(in, e.M, v) : 0.0;
        for (int o = 16; o > 0; o >>= 1)
            l += __shfl_xor_sync(0xffffffffu, l, o);
        if ((m & 31) == 0 && live)
            e.loss_part[m >> 5] = l;
    }
    if ((e.out_h || e.out_ht) && live)
        store_bf16(e, m, n, v);
}

// Bias gradient db[n] = sum_b dt[n][b] over the transposed bfloat16 gradient:
// BIAS_ROWS values per warp, each lane-strided FP32 partial sums, then a fixed
// shuffle tree.
constexpr int BIAS_ROWS = 2, BIAS_CTA_ROWS = BIAS_ROWS * GB_THREADS / 32;
__device__ __forceinline__ void bias_gradient(const GemmArgs &a, int cta)
{
    const int lane = threadIdx.x & 31;
    const int n0 = cta * BIAS_CTA_ROWS + (threadIdx.x >> 5) * BIAS_ROWS;
    float s[BIAS_ROWS];
#pragma unroll
    for (int i = 0; i < BIAS_ROWS; ++i)
        s[i] = 0.f;
#pragma unroll 4
    for (int b = lane; b < a.bias_b; b += 32)
#pragma unroll
        for (int i = 0; i < BIAS_ROWS; ++i)
            if (n0 + i < a.bias_n)
                s[i] += __bfloat162float(a.bias_dt[(size_t)(n0 + i) * a.bias_b + b]);
#pragma unroll
    for (int i = 0; i < BIAS_ROWS; ++i) {
        for (int o = 16; o > 0; o >>= 1)
            s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
        if (lane == 0 && n0 + i < a.bias_n)
            a.bias_db[n0 + i] = s[i];
    }
}

// Batch loss from the sums of 32 rows, in their order (at most 32 of them).
__device__ __forceinline__ void loss_total(const GemmArgs &a)
{
    if (threadIdx.x >= 32)
        return;
    const int n = (a.loss_rows + 31) / 32;
    const double v = (int)threadIdx.x < n ? a.loss_part[threadIdx.x] : 0.0;
    double t = 0.0;
    for (int w = 0; w < n; ++w)
        t += __shfl_sync(0xffffffffu, v, w);
    if (threadIdx.x == 0)
        a.loss[0] = (float)(t / a.loss_rows);
}

// ------------------------------------------------------------------ the GEMM
__global__ void __launch_bounds__(GB_THREADS, 2) umma_gemm_kernel(const __grid_constant__ GemmArgs args)
{
    int tile = blockIdx.x;
    if (tile >= args.tiles[0] + args.tiles[1]) {
        tile -= args.tiles[0] + args.tiles[1];
        grid_wait();
        grid_release();
        if (tile * BIAS_CTA_ROWS < args.bias_n)
            bias_gradient(args, tile);
        else
            loss_total(args);
        return;
    }
    const int p = tile >= args.tiles[0] ? 1 : 0;
    tile -= p ? args.tiles[0] : 0;
    const GemmEpi &e = args.e[p];
    const CUtensorMap *tmA = &args.ta[p], *tmB = &args.tb[p];
    extern __shared__ uint8_t gsm_raw[];
    const uint32_t raw = smem_u32(gsm_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *gsm = gsm_raw + (base - raw);
    const uint32_t bar_full = base + GB_BAR_OFF;
    const uint32_t bar_empty = bar_full + 8 * GB_STAGES;
    const uint32_t bar_done = bar_empty + 8 * GB_STAGES;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(gsm + GB_BAR_OFF + 16 * GB_STAGES + 8);
    volatile int *s_fail = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m_tiles = (e.M + GB_M - 1) / GB_M;
    const int m0 = tile % m_tiles * GB_M, n0 = tile / m_tiles * GB_N;
    const int nk = (e.K + GB_K - 1) / GB_K;

    if (threadIdx.x == 0) {
        for (int s = 0; s < GB_STAGES; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        mbar_init(bar_done, 1);
        *s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(GB_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_wait();
    grid_release();

    if (warp == 0) {
        if (lane == 0) {  // TMA producer
            int last[GB_STAGES];
            for (int s = 0; s < GB_STAGES; ++s)
                last[s] = -1;
            for (int kb = 0; kb < nk; ++kb) {
                const int s = kb % GB_STAGES;
                if (kb >= GB_STAGES && !mbar_wait(bar_empty + 8 * s, ((kb / GB_STAGES) - 1) & 1, e.timeout_ns)) {
                    *s_fail = 1;
                    break;
                }
                mbar_expect_tx(bar_full + 8 * s, (uint32_t)GB_STAGE);  // a box counts in full, zero fill included
                const uint32_t a = base + s * GB_STAGE;
                tma_load_2d(a, tmA, kb * GB_K, m0, bar_full + 8 * s);
                tma_load_2d(a + GB_TILE_A, tmB, kb * GB_K, n0, bar_full + 8 * s);
                last[s] = kb;
            }
            // no copy may still be landing when the CTA leaves
            for (int s = 0; s < GB_STAGES; ++s)
                if (last[s] >= 0 && !mbar_wait(bar_full + 8 * s, (last[s] / GB_STAGES) & 1, e.timeout_ns))
                    *s_fail = 1;
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) {  // MMA issuer
            for (int kb = 0; kb < nk; ++kb) {
                const int s = kb % GB_STAGES;
                if (!mbar_wait(bar_full + 8 * s, (kb / GB_STAGES) & 1, e.timeout_ns)) {
                    *s_fail = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t a = base + s * GB_STAGE, b = a + GB_TILE_A;
                const int steps = slab_steps(e.K, kb);
                for (int j = 0; j < steps; ++j)
                    umma_bf16(tmem, smem_desc(a + 32 * j), smem_desc(b + 32 * j), (kb | j) != 0 ? 1u : 0u);
                umma_commit(bar_empty + 8 * s);
            }
            umma_commit(bar_done);  // arrives once every MMA issued above has completed
        }
        __syncwarp();
    }

    // epilogue: every warp drains its own 32 TMEM lanes
    const int m = m0 + warp * 32 + lane;
    EpiInputs in;
    epi_fetch(e, m, n0, in);
    const int ok = __syncthreads_and(mbar_wait(bar_done, 0, e.timeout_ns) ? 1 : 0) && !*s_fail;
    tc_fence_after();
    if (ok) {
        const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll
        for (int nc = 0; nc < GB_N; nc += 16) {
            if (n0 + nc < e.N) {
                float v[16];
                tmem_ld16(trow + (uint32_t)nc, v);
                epi_store(e, m, n0 + nc, nc, in, v);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(GB_TMEM_COLS)
                     : "memory");
    }
    if (threadIdx.x == 0 && !ok)
        atomicCAS(e.err, 0, RF_ERR_TIMEOUT);
}

// ------------------------------------------------------------------ a few rows at once
// Forward pass of up to SMALL_BATCH rows (a frame's proposal is one) in one launch: a
// cluster of 8 CTAs x 16 warps, each warp two outputs of every layer, each CTA 32
// outputs of a hidden layer.  A lane takes every 32nd 16-byte piece of its warp's weight
// rows and loads those of all layers before it starts, so the 0.7 MB of weights cross
// once and at once; FP32 partial sums, a fixed shuffle tree, activations rounded to
// bfloat16 as the products' epilogue does and written to all CTAs' shared memory between
// cluster barriers.  Bound by latency: four dependent layers of a load, a sum and a
// barrier, and one row's sums after another's.  Against the four chained products:
// 6.4 : 20.7 us back to back at 1 row (4.4 of device time), 12.4 : 20.7 at 8.  A row more
// costs 0.9 us, so the two would meet near 16 rows; 8 is as many as a frame or a last batch
// asks for with rows and activations in 26 KB of static shared memory (16 need 51 of 48).
constexpr int SMALL_BATCH = 8, SMALL_CTAS = 8, SMALL_THREADS = 512;
constexpr int SMALL_PIECES = (RF_MLP_IN / 8 + 31) / 32;  // 16-byte pieces of a first-layer row per lane
static_assert(SMALL_CTAS * SMALL_THREADS / 32 * 2 == RF_MLP_HIDDEN && RF_MLP_HIDDEN == 256, "two outputs per warp");
static_assert(RF_MLP_OUT == 2 * SMALL_CTAS, "a warp of each CTA for the outputs");

struct SmallArgs {
    const bf16 *x, *w[4];
    const float *bias[4];
    float *out;
    int B;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// s += sum of the 8 products of two 16-byte pieces
__device__ __forceinline__ float dot8(const uint4 &a, const uint4 &b, float s)
{
    const uint32_t p[4] = {a.x, a.y, a.z, a.w}, q[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // a bfloat16 is the upper half of an FP32
        s = fmaf(__uint_as_float(p[i] << 16), __uint_as_float(q[i] << 16), s);
        s = fmaf(__uint_as_float(p[i] & 0xffff0000u), __uint_as_float(q[i] & 0xffff0000u), s);
    }
    return s;
}

// Two outputs of the warp for row `in` (16-byte pieces in shared memory), in every lane.
template <int PIECES>
__device__ __forceinline__ float2 dot_rows(const uint4 (&w)[2][PIECES], const uint4 *in, int pieces, float2 bias)
{
    const int lane = threadIdx.x & 31;
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int i = 0; i < PIECES; ++i)
        if (lane + 32 * i < pieces) {
            const uint4 v = in[lane + 32 * i];
            s0 = dot8(w[0][i], v, s0);
            s1 = dot8(w[1][i], v, s1);
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    return make_float2(s0 + bias.x, s1 + bias.y);
}

// Rectified, rounded outputs n, n + 1 of row b into the `h` of all CTAs (lane r: CTA r).
__device__ __forceinline__ void share_pair(const uint4 *h, int b, int n, float2 v)
{
    const uint32_t lane = threadIdx.x & 31;
    const __nv_bfloat162 q = __floats2bfloat162_rn(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f));
    uint32_t bits, dst;
    memcpy(&bits, &q, sizeof bits);
    const uint32_t own = smem_u32(h) + 2 * (b * RF_MLP_HIDDEN + n);
    if (lane < SMALL_CTAS) {
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(own), "r"(lane));
        asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(dst), "r"(bits) : "memory");
    }
}

__global__ void __cluster_dims__(SMALL_CTAS, 1, 1) __launch_bounds__(SMALL_THREADS, 1)
    forward_small_kernel(const SmallArgs a)
{
    constexpr int XP = RF_MLP_IN / 8, HP = RF_MLP_HIDDEN / 8;  // pieces of a row
    __shared__ uint4 x[SMALL_BATCH * XP];
    __shared__ uint4 h[3][SMALL_BATCH * HP];
    cluster_arrive();  // with the wait below: every CTA runs before another writes to it
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cta = blockIdx.x;
    const int n = (cta * (SMALL_THREADS / 32) + warp) * 2;     // the warp's hidden outputs n, n + 1
    uint4 w0[2][SMALL_PIECES], wh[2][2][1], w3[2][1];
    float2 bias[4];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
#pragma unroll
        for (int i = 0; i < SMALL_PIECES; ++i)
            w0[r][i] = lane + 32 * i < XP ? __ldg(reinterpret_cast<const uint4 *>(a.w[0]) + (n + r) * XP + lane + 32 * i)
                                          : make_uint4(0, 0, 0, 0);
        wh[0][r][0] = __ldg(reinterpret_cast<const uint4 *>(a.w[1]) + (n + r) * HP + lane);
        wh[1][r][0] = __ldg(reinterpret_cast<const uint4 *>(a.w[2]) + (n + r) * HP + lane);
        w3[r][0] = __ldg(reinterpret_cast<const uint4 *>(a.w[3]) + (2 * cta + r) * HP + lane);
    }
#pragma unroll
    for (int l = 0; l < 4; ++l)
        bias[l] = __ldg(reinterpret_cast<const float2 *>(a.bias[l] + (l < 3 ? n : 2 * cta)));
    for (int i = threadIdx.x; i < a.B * XP; i += SMALL_THREADS)
        x[i] = __ldg(reinterpret_cast<const uint4 *>(a.x) + i);
    __syncthreads();
    cluster_wait();
    for (int b = 0; b < a.B; ++b)
        share_pair(h[0], b, n, dot_rows(w0, x + b * XP, XP, bias[0]));
#pragma unroll
    for (int l = 0; l < 2; ++l) {
        cluster_arrive();
        cluster_wait();
        for (int b = 0; b < a.B; ++b)
            share_pair(h[l + 1], b, n, dot_rows(wh[l], h[l] + b * HP, HP, bias[l + 1]));
    }
    cluster_arrive();
    cluster_wait();
    for (int b = warp; b < a.B; b += SMALL_THREADS / 32) {
        const float2 o = dot_rows(w3, h[2] + b * HP, HP, bias[3]);
        if (lane < 2)
            a.out[b * RF_MLP_OUT + 2 * cta + lane] = lane ? o.y : o.x;
    }
}

// ------------------------------------------------------------------ elementwise kernels
// Layout of the flat FP32 parameter vector (W1, b1, W2, b2, W3, b3, W4, b4; each W
// row-major out x in) and of the packed bfloat16 weight copies (W_l at pk_off[l],
// its transpose at the same offset of the transposed copy).
struct LayerTable {
    int w_off[4], pk_off[4], out[4], in[4];
    int total;
};

__device__ __forceinline__ int layer_of(const LayerTable &L, int p)
{
    int l = 0;
    while (l < 3 && p >= L.w_off[l + 1])
        ++l;
    return l;
}

// Adam (Kingma & Ba 2015, Algorithm 1) on the FP32 parameters when `update`,
// then the bfloat16 weights the GEMMs read, row-major and transposed.
__global__ void adam_kernel(float *theta, const float *grad, float *m, float *v, const LayerTable L, float lr,
                            float b1, float b2, float eps, float bc1, float bc2, int update, bf16 *w, bf16 *wt)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < L.total; p += gridDim.x * blockDim.x) {
        float th = theta[p];
        if (update) {
            const float g = grad[p];
            const float mm = b1 * m[p] + (1.f - b1) * g;
            const float vv = b2 * v[p] + (1.f - b2) * g * g;
            m[p] = mm;
            v[p] = vv;
            th -= lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
            theta[p] = th;
        }
        const int l = layer_of(L, p);
        const int q = p - L.w_off[l];
        if (q < L.out[l] * L.in[l]) {
            const int o = q / L.in[l], i = q - o * L.in[l];
            const bf16 h = __float2bfloat16_rn(th);
            w[L.pk_off[l] + q] = h;
            wt[L.pk_off[l] + i * L.out[l] + o] = h;
        }
    }
}

// Rows idx[b] (row b when idx is NULL) of a dataset into the batch buffers: the
// input row-major and, when xt is given (B then a multiple of 8), transposed, the
// target.  Out-of-range rows raise RF_ERR_ARG and are skipped.  A CTA moves 32 rows x
// 64 columns through shared memory, so both copies are written 16 bytes at a time
// (one CTA per row stored the transpose 2 bytes at a time, 8 us of a 512-row batch
// under the profiler); it reads 16 bytes at a time when the dataset is so aligned.
constexpr int GATHER_ROWS = 32, GATHER_COLS = 64, GATHER_THREADS = GATHER_ROWS * GATHER_COLS / 8;
static_assert(RF_MLP_IN % GATHER_COLS == 0, "whole column blocks");
__global__ void __launch_bounds__(GATHER_THREADS) gather_kernel(const bf16 *x_all, const float *y_all, const int *idx,
                                                                int n_all, int B, bf16 *x, bf16 *xt, float *y,
                                                                int *err)
{
    __shared__ uint32_t tile[GATHER_ROWS][GATHER_COLS / 2 + 1];
    __shared__ uint8_t valid[GATHER_ROWS];
    grid_release();
    const int b0 = blockIdx.x * GATHER_ROWS, k0 = blockIdx.y * GATHER_COLS;
    {
        const int row = threadIdx.x >> 3, c = threadIdx.x & 7, b = b0 + row;
        const int r = b < B ? (idx ? __ldg(&idx[b]) : b) : -1;
        const bool in = r >= 0 && r < n_all;
        if (b < B && !in && c == 0)
            atomicCAS(err, 0, RF_ERR_ARG);
        if (c == 0)
            valid[row] = in;
        if (in) {
            const bf16 *src = x_all + (size_t)r * RF_MLP_IN + k0 + 8 * c;
            uint4 q;
            if (((uintptr_t)x_all & 15) == 0) {
                q = __ldg(reinterpret_cast<const uint4 *>(src));
            } else {
                bf16 h[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    h[i] = src[i];
                memcpy(&q, h, sizeof q);
            }
            *reinterpret_cast<uint4 *>(x + (size_t)b * RF_MLP_IN + k0 + 8 * c) = q;
            tile[row][4 * c] = q.x;
            tile[row][4 * c + 1] = q.y;
            tile[row][4 * c + 2] = q.z;
            tile[row][4 * c + 3] = q.w;
        }
        if (blockIdx.y == 0 && c < 6 && in)
            y[b * 6 + c] = y_all[(size_t)r * 6 + c];
    }
    if (!xt)
        return;
    __syncthreads();
    const int k = threadIdx.x >> 2, row = (threadIdx.x & 3) * 8, b = b0 + row;
    if (b >= B)
        return;
    bf16 h[8];
    bool all = true;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        h[i] = reinterpret_cast<const bf16 *>(tile[row + i])[k];
        all = all && valid[row + i];
    }
    bf16 *o = xt + (size_t)(k0 + k) * B + b;
    if (all) {
        uint4 q;
        memcpy(&q, h, sizeof q);
        *reinterpret_cast<uint4 *>(o) = q;
    } else {
        for (int i = 0; i < 8; ++i)
            if (valid[row + i])
                o[i] = h[i];
    }
}

// ------------------------------------------------------------------ host: tensor maps and launches
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

rf_status tensor_map_encoder(EncodeTiledFn *out)
{
    static std::mutex mu;
    static EncodeTiledFn fn = nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !p) {
            set_error("cuTensorMapEncodeTiled not available (%s)", cudaGetErrorString(e));
            return RF_ERR_CUDA;
        }
        fn = (EncodeTiledFn)p;
    }
    *out = fn;
    return RF_OK;
}

// TMA map of a row-major bfloat16 operand [rows x cols] with leading dimension ld:
// box of 64 columns (128 B) x box_rows rows, 128-byte swizzle; reads past rows or
// cols fill 0.
rf_status operand_map(CUtensorMap *map, const bf16 *ptr, int rows, int cols, int ld, int box_rows)
{
    RF_CHECK_ARG(ptr && ((uintptr_t)ptr & 15) == 0, "operand not 16-byte aligned");
    RF_CHECK_ARG(rows >= 1 && cols >= 1 && ld >= cols && ld % 8 == 0, "operand shape");
    EncodeTiledFn enc;
    rf_status st = tensor_map_encoder(&enc);
    if (st != RF_OK)
        return st;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * sizeof(bf16)};
    const cuuint32_t box[2] = {(cuuint32_t)GB_K, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(ptr), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        set_error("cuTensorMapEncodeTiled failed (%d)", (int)r);
        return RF_ERR_CUDA;
    }
    return RF_OK;
}

rf_status gemm_smem_attr()
{
    static std::mutex mu;
    static unsigned long long done_mask = 0;
    int dev = 0;
    RF_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 64 && !(done_mask >> dev & 1ull)) {
        RF_CUDA(cudaFuncSetAttribute(umma_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, GB_SMEM));
        done_mask |= 1ull << dev;
    }
    return RF_OK;
}

// Product p of a launch: C = A . B^T with the epilogue of e (e.M, e.N, e.K set by
// the caller).
rf_status gemm_add(GemmArgs &a, int p, const bf16 *A, int lda, const bf16 *B, int ldb, const GemmEpi &e)
{
    RF_CHECK_ARG(e.M >= 1 && e.N >= 1 && e.N % 16 == 0 && e.K >= 1, "product shape");
    RF_CHECK_ARG(!e.out_h || e.ld_h % 8 == 0, "ld_h");
    RF_CHECK_ARG(!e.out_f || e.ld_f % 4 == 0, "ld_f");
    rf_status st = operand_map(&a.ta[p], A, e.M, e.K, lda, GB_M);
    if (st == RF_OK)
        st = operand_map(&a.tb[p], B, e.N, e.K, ldb, GB_N);
    a.e[p] = e;
    a.tiles[p] = ((e.M + GB_M - 1) / GB_M) * ((e.N + GB_N - 1) / GB_N);
    return st;
}

// `chained`: the launch before on this stream is a kernel of this file that releases
// its dependents, so this one's setup may overlap its end.
rf_status gemm_launch(const GemmArgs &a, bool chained, cudaStream_t s)
{
    rf_status st = gemm_smem_attr();
    if (st != RF_OK)
        return st;
    const int grid = a.tiles[0] + a.tiles[1] + (a.bias_n + BIAS_CTA_ROWS - 1) / BIAS_CTA_ROWS + (a.loss ? 1 : 0);
    RF_CUDA(launch_chained(chained, umma_gemm_kernel, grid, GB_THREADS, GB_SMEM, s, a));
    return RF_OK;
}

void gather(const bf16 *x_all, const float *y_all, const int *idx, int n_all, int B, bf16 *x, bf16 *xt, float *y,
            int *err, cudaStream_t s)
{
    const dim3 grid((B + GATHER_ROWS - 1) / GATHER_ROWS, RF_MLP_IN / GATHER_COLS);
    gather_kernel<<<grid, GATHER_THREADS, 0, s>>>(x_all, y_all, idx, n_all, B, x, xt, y, err);
}

GemmEpi epi(int M, int N, int K, int mode, int *err, long long timeout_ns)
{
    GemmEpi e;
    memset(&e, 0, sizeof e);
    e.M = M;
    e.N = N;
    e.K = K;
    e.mode = mode;
    e.err = err;
    e.timeout_ns = timeout_ns;
    return e;
}

}  // namespace
// The quantities training selects and calibrates the network with, over B rows
// of a batch (outputs `out`, inputs `x`, targets `y`): mu = x_v + o_mu (x_v the
// previous-offset inputs), s = clamp(o_s, -6, 6), e = y - mu, and per row
// sum_d e_d^2, e_d^2 exp(-2 s_d), y_d^2 (13 values, FP64).  One CTA; thread t
// takes rows t, t + blockDim, ...; the per-thread sums are combined by a fixed
// shuffle tree and warp order, and thread 0 adds them to acc (the calls for the
// successive batches of a data set run in stream order, so the total is fixed).
constexpr int EVAL_STATS = 13;
__global__ void eval_kernel(const float *out, const bf16 *x, const float *y, int B, int row0, float *mu_out,
                            double *acc)
{
    __shared__ double red[EVAL_STATS][32];
    double loc[EVAL_STATS];
    for (int e = 0; e < EVAL_STATS; ++e)
        loc[e] = 0.0;
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        for (int d = 0; d < 6; ++d) {
            const float mu = out[b * RF_MLP_OUT + d] +
                             __bfloat162float(x[(size_t)b * RF_MLP_IN + RF_MLP_IN_USED - 6 + d]);
            const float s = fminf(fmaxf(out[b * RF_MLP_OUT + 6 + d], -6.f), 6.f);
            const double yd = (double)y[b * 6 + d];
            const double e = yd - (double)mu;
            loc[0] += e * e;
            loc[1 + d] += e * e * exp(-2.0 * (double)s);
            loc[7 + d] += yd * yd;
            if (mu_out)
                mu_out[(size_t)(row0 + b) * 6 + d] = mu;
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int e = 0; e < EVAL_STATS; ++e) {
        double v = loc[e];
        for (int o = 16; o > 0; o >>= 1)
            v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0)
            red[e][w] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int e = 0; e < EVAL_STATS; ++e) {
            double t = 0.0;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q)
                t += red[e][q];
            acc[e] += t;
        }
}

__global__ void eval_finish_kernel(const double *acc, int n_rows, double *stats)
{
    if (threadIdx.x < EVAL_STATS)
        stats[threadIdx.x] = acc[threadIdx.x] / (double)n_rows;
}

// log k_d added to the output bias of the log-scale s_d, k_d^2 = stats[1 + d].
__global__ void calibrate_kernel(const double *stats, float *bias_s, float *k_out)
{
    const int d = threadIdx.x;
    if (d < 6) {
        const double k = sqrt(fmax(stats[1 + d], 1e-12));
        bias_s[d] += (float)log(k);
        k_out[d] = (float)k;
    }
}

}  // namespace rf

using namespace rf;

// ------------------------------------------------------------------ network handle
struct rf_mlp_s {
    int max_batch;
    LayerTable L;
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    bf16 *w = nullptr, *wt = nullptr;  // packed bfloat16 weights and transposes
    bf16 *x = nullptr, *xt = nullptr;
    bf16 *h[3] = {}, *ht[3] = {};      // hidden activations h1..h3 (row-major, transposed)
    bf16 *d[3] = {}, *dt[3] = {};      // masked hidden gradients
    bf16 *g = nullptr, *gt = nullptr;  // output gradients
    float *out = nullptr, *y = nullptr, *loss = nullptr;
    double *loss_part = nullptr;       // loss sums of 32 rows each
    double *eval_acc = nullptr;  // rf_mlp_evaluate: running sums, then the means (2 x EVAL_STATS)
    float *eval_k = nullptr;     // rf_mlp_calibrate_scale: k (6)
    int *err = nullptr;
    int step = 0;
    long long timeout_ns = 1000000000ll;
    std::vector<void *> allocs;
};

static const int kOut[4] = {RF_MLP_HIDDEN, RF_MLP_HIDDEN, RF_MLP_HIDDEN, RF_MLP_OUT};
static const int kIn[4] = {RF_MLP_IN, RF_MLP_HIDDEN, RF_MLP_HIDDEN, RF_MLP_HIDDEN};

static LayerTable layer_table()
{
    LayerTable L;
    int p = 0, k = 0;
    for (int l = 0; l < 4; ++l) {
        L.out[l] = kOut[l];
        L.in[l] = kIn[l];
        L.w_off[l] = p;
        L.pk_off[l] = k;
        p += kOut[l] * kIn[l] + kOut[l];
        k += kOut[l] * kIn[l];
    }
    L.total = p;
    return L;
}

static rf_status mlp_alloc(rf_mlp m, void **p, size_t bytes)
{
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess)
        return cuda_fail(e, "cudaMalloc(mlp)");
    m->allocs.push_back(*p);
    return RF_OK;
}

// Refresh the bfloat16 weight copies (update = 0) or take one Adam step.
static rf_status mlp_adam(rf_mlp m, int update, float lr, cudaStream_t s)
{
    const double b1 = 0.9, b2 = 0.999;
    float bc1 = 1.f, bc2 = 1.f;
    if (update) {
        m->step += 1;
        bc1 = (float)(1.0 - pow(b1, m->step));
        bc2 = (float)(1.0 - pow(b2, m->step));
    }
    adam_kernel<<<304, 256, 0, s>>>(m->theta, m->grad, m->m, m->v, m->L, lr, (float)b1, (float)b2, 1e-8f, bc1, bc2,
                                    update, m->w, m->wt);
    RF_CUDA(cudaGetLastError());
    return RF_OK;
}

// What a training forward pass leaves for the backward one.
struct TrainOut {
    float *out;   // outputs (B x 16)
    float *grad;  // flat gradient
    float *loss;
};

// Forward pass of B rows of x: hidden activations to m->h, outputs to out (B x 16,
// FP32).  With `train`, also the transposed activations, the outputs' gradient and the
// loss sums (x is then m->x).  `chained`: the rows come from a gather just launched.
static rf_status mlp_forward(rf_mlp m, const bf16 *x, int B, float *out, bool train, bool chained, cudaStream_t s)
{
    const LayerTable &L = m->L;
    if (!train && B <= SMALL_BATCH) {
        RF_CHECK_ARG(((uintptr_t)x & 15) == 0, "operand not 16-byte aligned");
        SmallArgs a;
        for (int l = 0; l < 4; ++l) {
            a.w[l] = m->w + L.pk_off[l];
            a.bias[l] = m->theta + L.w_off[l] + L.out[l] * L.in[l];
        }
        a.x = x;
        a.out = out;
        a.B = B;
        forward_small_kernel<<<SMALL_CTAS, SMALL_THREADS, 0, s>>>(a);
        RF_CUDA(cudaGetLastError());
        return RF_OK;
    }
    const bf16 *in = x;
    int ld_in = RF_MLP_IN;
    for (int l = 0; l < 4; ++l) {
        GemmEpi e = epi(B, L.out[l], L.in[l], l < 3 ? EPI_BIAS_RELU : (train ? EPI_LOSS : EPI_BIAS), m->err,
                        m->timeout_ns);
        e.bias = m->theta + L.w_off[l] + L.out[l] * L.in[l];
        if (l < 3 || train) {
            e.out_h = l < 3 ? m->h[l] : m->g;
            e.ld_h = L.out[l];
        }
        if (train) {
            e.out_ht = l < 3 ? m->ht[l] : m->gt;
            e.ld_ht = B;
        }
        if (l == 3) {
            e.out_f = out;
            e.ld_f = RF_MLP_OUT;
            e.x = x;
            e.y = m->y;
            e.loss_part = m->loss_part;
        }
        GemmArgs a;
        memset(&a, 0, sizeof a);
        rf_status st = gemm_add(a, 0, in, ld_in, m->w + L.pk_off[l], L.in[l], e);
        if (st == RF_OK)
            st = gemm_launch(a, chained || l > 0, s);
        if (st != RF_OK)
            return st;
        in = m->h[l < 3 ? l : 2];
        ld_in = RF_MLP_HIDDEN;
    }
    return RF_OK;
}

// Gather, forward, loss and backward of one batch.  A layer's weight, bias and input
// gradients read the same gradient of its outputs and are one launch, the loss and its
// gradient are the epilogue of the last forward product, and the launches are chained
// by programmatic dependent launch: 9 instead of 17 (and 3 copies of the results),
// 49 us instead of 146 us at 512 rows.
static rf_status mlp_gradient(rf_mlp m, const bf16 *x_all, const float *y_all, const int *idx, int n_all, int B,
                              const TrainOut &t, cudaStream_t s)
{
    const LayerTable &L = m->L;
    gather(x_all, y_all, idx, n_all, B, m->x, m->xt, m->y, m->err, s);
    RF_CUDA(cudaGetLastError());
    rf_status st = mlp_forward(m, m->x, B, t.out, true, true, s);
    if (st != RF_OK)
        return st;
    // layer 4: dW4 = g^T h3, db4 = sum_b g, dH3 = g W4 masked by h3 > 0
    const bf16 *dA = m->g, *dAt = m->gt;
    for (int l = 3; l >= 0; --l) {
        const bf16 *act_t = l > 0 ? m->ht[l - 1] : m->xt;  // the layer's input, transposed
        GemmArgs a;
        memset(&a, 0, sizeof a);
        GemmEpi e = epi(L.out[l], L.in[l], B, EPI_PLAIN, m->err, m->timeout_ns);
        e.out_f = t.grad + L.w_off[l];
        e.ld_f = L.in[l];
        st = gemm_add(a, 0, dAt, B, act_t, B, e);
        if (st != RF_OK)
            return st;
        a.bias_dt = dAt;
        a.bias_db = t.grad + L.w_off[l] + L.out[l] * L.in[l];
        a.bias_n = L.out[l];
        a.bias_b = B;
        if (l == 3) {
            a.loss_part = m->loss_part;
            a.loss = t.loss;
            a.loss_rows = B;
        }
        if (l > 0) {
            GemmEpi eb = epi(B, L.in[l], L.out[l], EPI_MASK, m->err, m->timeout_ns);
            eb.mask = m->h[l - 1];
            eb.ld_mask = RF_MLP_HIDDEN;
            eb.out_h = m->d[l - 1];
            eb.ld_h = RF_MLP_HIDDEN;
            eb.out_ht = m->dt[l - 1];
            eb.ld_ht = B;
            st = gemm_add(a, 1, dA, L.out[l], m->wt + L.pk_off[l], L.out[l], eb);
            if (st != RF_OK)
                return st;
            dA = m->d[l - 1];
            dAt = m->dt[l - 1];
        }
        st = gemm_launch(a, true, s);
        if (st != RF_OK)
            return st;
    }
    return RF_OK;
}

extern "C" {

int rf_mlp_num_params(void) { return layer_table().total; }

rf_status rf_mlp_create(int max_batch, rf_mlp *out)
{
    RF_CHECK_ARG(out != nullptr, "null output");
    *out = nullptr;
    RF_CHECK_ARG(max_batch >= 1 && max_batch <= RF_MLP_MAX_BATCH, "max_batch outside [1, RF_MLP_MAX_BATCH]");
    rf_mlp m = new rf_mlp_s();
    m->max_batch = (max_batch + 7) / 8 * 8;
    m->L = layer_table();
    const size_t P = (size_t)m->L.total, PK = (size_t)m->L.pk_off[3] + (size_t)RF_MLP_OUT * RF_MLP_HIDDEN;
    const size_t Bc = (size_t)m->max_batch;
    rf_status st = RF_OK;
    void **fl[4] = {(void **)&m->theta, (void **)&m->grad, (void **)&m->m, (void **)&m->v};
    for (int i = 0; i < 4 && st == RF_OK; ++i)
        st = mlp_alloc(m, fl[i], P * sizeof(float));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->w, PK * sizeof(bf16));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->wt, PK * sizeof(bf16));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->x, Bc * RF_MLP_IN * sizeof(bf16));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->xt, Bc * RF_MLP_IN * sizeof(bf16));
    for (int l = 0; l < 3 && st == RF_OK; ++l) {
        st = mlp_alloc(m, (void **)&m->h[l], Bc * RF_MLP_HIDDEN * sizeof(bf16));
        if (st == RF_OK)
            st = mlp_alloc(m, (void **)&m->ht[l], Bc * RF_MLP_HIDDEN * sizeof(bf16));
        if (st == RF_OK)
            st = mlp_alloc(m, (void **)&m->d[l], Bc * RF_MLP_HIDDEN * sizeof(bf16));
        if (st == RF_OK)
            st = mlp_alloc(m, (void **)&m->dt[l], Bc * RF_MLP_HIDDEN * sizeof(bf16));
    }
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->g, Bc * RF_MLP_OUT * sizeof(bf16));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->gt, Bc * RF_MLP_OUT * sizeof(bf16));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->out, Bc * RF_MLP_OUT * sizeof(float));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->y, Bc * 6 * sizeof(float));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->loss, sizeof(float));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->loss_part, (RF_MLP_MAX_TRAIN_BATCH / 32) * sizeof(double));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->err, sizeof(int));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->eval_acc, 2 * EVAL_STATS * sizeof(double));
    if (st == RF_OK)
        st = mlp_alloc(m, (void **)&m->eval_k, 6 * sizeof(float));
    if (st == RF_OK) {
        cudaError_t e = cudaMemset(m->theta, 0, P * sizeof(float));
        if (e == cudaSuccess)
            e = cudaMemset(m->grad, 0, P * sizeof(float));
        if (e == cudaSuccess)
            e = cudaMemset(m->m, 0, P * sizeof(float));
        if (e == cudaSuccess)
            e = cudaMemset(m->v, 0, P * sizeof(float));
        if (e == cudaSuccess)
            e = cudaMemset(m->w, 0, PK * sizeof(bf16));
        if (e == cudaSuccess)
            e = cudaMemset(m->wt, 0, PK * sizeof(bf16));
        if (e == cudaSuccess)
            e = cudaMemset(m->err, 0, sizeof(int));
        if (e != cudaSuccess)
            st = cuda_fail(e, "cudaMemset(mlp)");
    }
    // resolve the tensor-map encoder and the kernel's shared-memory limit now, so
    // that no later call (for example inside a stream capture) does it first
    EncodeTiledFn enc;
    if (st == RF_OK)
        st = tensor_map_encoder(&enc);
    if (st == RF_OK)
        st = gemm_smem_attr();
    if (st != RF_OK) {
        rf_mlp_destroy(m);
        return st;
    }
    *out = m;
    return RF_OK;
}

void rf_mlp_destroy(rf_mlp m)
{
    if (!m)
        return;
    for (void *p : m->allocs)
        cudaFree(p);
    delete m;
}

rf_status rf_mlp_set_params(rf_mlp m, const float *theta_host)
{
    RF_CHECK_ARG(m && theta_host, "null pointer");
    const size_t P = (size_t)m->L.total;
    RF_CUDA(cudaMemcpy(m->theta, theta_host, P * sizeof(float), cudaMemcpyHostToDevice));
    RF_CUDA(cudaMemset(m->m, 0, P * sizeof(float)));
    RF_CUDA(cudaMemset(m->v, 0, P * sizeof(float)));
    m->step = 0;
    rf_status st = mlp_adam(m, 0, 0.f, 0);
    if (st != RF_OK)
        return st;
    RF_CUDA(cudaDeviceSynchronize());
    return RF_OK;
}

rf_status rf_mlp_get_params(rf_mlp m, float *theta_host)
{
    RF_CHECK_ARG(m && theta_host, "null pointer");
    RF_CUDA(cudaDeviceSynchronize());
    RF_CUDA(cudaMemcpy(theta_host, m->theta, (size_t)m->L.total * sizeof(float), cudaMemcpyDeviceToHost));
    return RF_OK;
}

rf_status rf_mlp_forward(rf_mlp m, const uint16_t *x_dev, int batch, float *out_dev, void *stream)
{
    RF_CHECK_ARG(m && x_dev && out_dev, "null pointer");
    RF_CHECK_ARG(batch >= 1 && batch <= m->max_batch, "batch outside [1, max_batch]");
    return mlp_forward(m, reinterpret_cast<const bf16 *>(x_dev), batch, out_dev, false, false, (cudaStream_t)stream);
}

rf_status rf_mlp_gradient(rf_mlp m, const uint16_t *x_all_dev, const float *y_all_dev, const int *idx_dev, int n_all,
                          int batch, float *grad_dev, float *loss_dev, float *out_dev, void *stream)
{
    RF_CHECK_ARG(m && x_all_dev && y_all_dev, "null pointer");
    RF_CHECK_ARG(batch >= 8 && batch <= m->max_batch && batch % 8 == 0 && batch <= RF_MLP_MAX_TRAIN_BATCH,
                 "training batch must be a multiple of 8 in [8, min(max_batch, RF_MLP_MAX_TRAIN_BATCH)]");
    RF_CHECK_ARG(n_all >= 1 && (idx_dev || n_all >= batch), "dataset rows");
    cudaStream_t s = (cudaStream_t)stream;
    // straight into the caller's buffers where the 16-byte stores allow it
    TrainOut t;
    t.out = out_dev && ((uintptr_t)out_dev & 15) == 0 ? out_dev : m->out;
    t.grad = grad_dev && ((uintptr_t)grad_dev & 15) == 0 ? grad_dev : m->grad;
    t.loss = loss_dev ? loss_dev : m->loss;
    rf_status st = mlp_gradient(m, reinterpret_cast<const bf16 *>(x_all_dev), y_all_dev, idx_dev, n_all, batch, t, s);
    if (st != RF_OK)
        return st;
    if (grad_dev && t.grad != grad_dev)
        RF_CUDA(cudaMemcpyAsync(grad_dev, t.grad, (size_t)m->L.total * sizeof(float), cudaMemcpyDeviceToDevice, s));
    if (out_dev && t.out != out_dev)
        RF_CUDA(cudaMemcpyAsync(out_dev, t.out, (size_t)batch * RF_MLP_OUT * sizeof(float), cudaMemcpyDeviceToDevice,
                                s));
    return RF_OK;
}

rf_status rf_mlp_train_step(rf_mlp m, const uint16_t *x_all_dev, const float *y_all_dev, const int *idx_dev, int n_all,
                            int batch, float lr, float *loss_dev, void *stream)
{
    rf_status st = rf_mlp_gradient(m, x_all_dev, y_all_dev, idx_dev, n_all, batch, nullptr, loss_dev, nullptr, stream);
    if (st != RF_OK)
        return st;
    RF_CHECK_ARG(lr >= 0.f, "negative learning rate");
    return mlp_adam(m, 1, lr, (cudaStream_t)stream);
}

rf_status rf_mlp_evaluate(rf_mlp m, const uint16_t *x_all_dev, const float *y_all_dev, const int *idx_dev,
                          int n_all, int n_rows, float *mu_dev, double *stats_dev, void *stream)
{
    RF_CHECK_ARG(m && x_all_dev && y_all_dev, "null pointer");
    RF_CHECK_ARG(n_rows >= 1 && n_all >= 1 && (idx_dev || n_rows <= n_all), "dataset rows");
    cudaStream_t s = (cudaStream_t)stream;
    RF_CUDA(cudaMemsetAsync(m->eval_acc, 0, EVAL_STATS * sizeof(double), s));
    const bf16 *x_all = reinterpret_cast<const bf16 *>(x_all_dev);
    for (int r0 = 0; r0 < n_rows; r0 += m->max_batch) {
        const int B = std::min(m->max_batch, n_rows - r0);
        // rows idx[r0 ..] (or r0 ..) into the batch buffers; no transposed copy is needed
        if (idx_dev)
            gather(x_all, y_all_dev, idx_dev + r0, n_all, B, m->x, nullptr, m->y, m->err, s);
        else
            gather(x_all + (size_t)r0 * RF_MLP_IN, y_all_dev + (size_t)r0 * 6, nullptr, n_all - r0, B, m->x, nullptr,
                   m->y, m->err, s);
        RF_CUDA(cudaGetLastError());
        rf_status st = mlp_forward(m, m->x, B, m->out, false, true, s);
        if (st != RF_OK)
            return st;
        eval_kernel<<<1, 256, 0, s>>>(m->out, m->x, m->y, B, r0, mu_dev, m->eval_acc);
        RF_CUDA(cudaGetLastError());
    }
    eval_finish_kernel<<<1, 32, 0, s>>>(m->eval_acc, n_rows, m->eval_acc + EVAL_STATS);
    RF_CUDA(cudaGetLastError());
    if (stats_dev)
        RF_CUDA(cudaMemcpyAsync(stats_dev, m->eval_acc + EVAL_STATS, EVAL_STATS * sizeof(double),
                                cudaMemcpyDeviceToDevice, s));
    return RF_OK;
}

rf_status rf_mlp_calibrate_scale(rf_mlp m, const uint16_t *x_all_dev, const float *y_all_dev, const int *idx_dev,
                                 int n_all, int n_rows, float k_host[6], void *stream)
{
    RF_CHECK_ARG(m && k_host, "null pointer");
    cudaStream_t s = (cudaStream_t)stream;
    rf_status st = rf_mlp_evaluate(m, x_all_dev, y_all_dev, idx_dev, n_all, n_rows, nullptr, nullptr, stream);
    if (st != RF_OK)
        return st;
    const LayerTable &L = m->L;
    float *b4 = m->theta + L.w_off[3] + L.out[3] * L.in[3];
    calibrate_kernel<<<1, 32, 0, s>>>(m->eval_acc + EVAL_STATS, b4 + 6, m->eval_k);
    RF_CUDA(cudaGetLastError());
    RF_CUDA(cudaMemcpyAsync(k_host, m->eval_k, 6 * sizeof(float), cudaMemcpyDeviceToHost, s));
    RF_CUDA(cudaStreamSynchronize(s));
    return RF_OK;
}

rf_status rf_mlp_status(rf_mlp m)
{
    RF_CHECK_ARG(m != nullptr, "null network");
    int h = 0;
    RF_CUDA(cudaDeviceSynchronize());
    RF_CUDA(cudaMemcpy(&h, m->err, sizeof(int), cudaMemcpyDeviceToHost));
    RF_CUDA(cudaMemset(m->err, 0, sizeof(int)));
    if (h != 0)
        set_error("rf_mlp: device status %d", h);
    return h;
}

}  // extern "C"
