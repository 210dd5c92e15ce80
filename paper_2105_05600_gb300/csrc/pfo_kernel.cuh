// pfo_kernel.cuh -- the persistent PFO kernel (Algorithm 1 for one frame of one or
// several sequences) and its launch descriptors, shared by the host code in pfo.cu
// and the per-storage-type translation units that instantiate the kernel
// (pfo_kernels_f32.cu, pfo_kernels_f16.cu, pfo_kernels_i16.cu, compiled in parallel).
#pragma once
#include <math.h>
#include <string.h>

#include <algorithm>

#include "fitness.cuh"

namespace rf {

constexpr int MAX_BATCH = RF_MAX_BATCH;
constexpr int MAX_LEVELS = RF_MAX_LEVELS;
// The fitness split of a sequence is computed for this warp count (not for the
// actual grid), so a sequence's results do not depend on the launch shape or on
// the other sequences of a batch.
constexpr int WORK_WARPS_DEFAULT = 3648;
constexpr int WORK_WARPS_MAX = 7296;

rf_status launch_integrate_dev(const VolumeDesc &V, const float *depth, const Intr &K, const float *pose_dev,
                               const int *status_dev, cudaStream_t s);

constexpr int SORT_BITS = 10;
constexpr int SORT_BUCKETS = 1 << SORT_BITS;
constexpr int SORT_BLOCK = 512;  // particles that one CTA ranks together
// Lookups an iteration (particles x points of the level) from which the scoring order pays
// for itself.  Frames of ten iterations with the order against without it, 64^3 float, 256^3
// and 512^3 int16 and 384^3 half maps, two rooms each, mean (range): 4.9 M lookups 0.990
// (0.97 .. 1.01) times as fast, 9.8 M 0.995, 14.7 M 0.993, 19.7 M 1.008 (0.97 .. 1.06),
// 39 M 1.014 (0.96 .. 1.07), 59 M 1.017 (0.99 .. 1.07): wide swarms gain, tight ones lose
// its 2 to 4 us an iteration, and the mean crosses 1 between 14.7 M and 19.7 M.
constexpr long long SORT_MIN_WORK = 1ll << 24;

// ------------------------------------------------------------------ launch descriptors
struct ProblemDesc {
    VolumeDesc V;
    Intr K;
    const float *depth, *prev_depth;
    const float *pst;  // template, structure of arrays, leading dimension n_tmpl
    int n_tmpl;
    int n_levels;
    int lvl_n[MAX_LEVELS], lvl_stride[MAX_LEVELS], lvl_nw[MAX_LEVELS], lvl_m[MAX_LEVELS], lvl_off[MAX_LEVELS];
    int m_all;  // points of all levels (concatenated in pts at lvl_off)
    const float *prev_pose;
    const float *init_pose;  // c_0 (NULL: prev_pose)
    const int *run_flag;     // NULL, or skip the frame when *run_flag == 0 at launch
    float *out_pose;
    rf_frame_stats *stats;
    float *scale;  // r_0 in, r_1 out
    float4 *pts, *cpts;
    double *part_S;
    int *part_n;
    int max_chunks;
    int *ord;  // [n_tmpl] particles in scoring order, rebuilt every iteration; ord[n_tmpl] = place of particle 0
    int *key;  // [n_tmpl] bucket | place among its block's particles of the bucket << SORT_BITS
    uint16_t *bucket_counts;  // [blocks of SORT_BLOCK particles][SORT_BUCKETS]
    int *status;
    float tau, beta, eps, stop_eps;
    int k_max, flags;
};

struct alignas(16) GridSync {
    unsigned int count;  // CTAs that have arrived, over all barriers of the launch
    int abort;
    int skip;  // test hook: block 0 leaves at the first barrier without arriving
};

struct BatchParams {
    ProblemDesc prob[MAX_BATCH];
    int B;
    int k_max_all;
    int work_warps;
    GridSync *gs;       // gs and unit_ctr are one allocation, zero at launch
    int *unit_ctr;      // [RF_MAX_ITERS]
    int *block_counts;  // [grid][MAX_BATCH]
    double *aps;        // [grid][MAX_BATCH][APW]
    long long timeout_ns;
};

// ------------------------------------------------------------------ grid barrier
// Counter barrier over all CTAs of the cooperative launch.  `count` only grows: the
// n-th barrier is open once it reaches n x gridDim, so an arrival is one release
// increment and a wait is one polled word -- no reset, no second flag to pass on
// and no back-off sleep (304 CTAs of a GB300, all arriving together: 1.5 to 2.1 us,
// against 2.3 to 2.9 us for a sense-reversing counter with a generation word).  Every
// wait is bounded: after timeout_ns the CTA sets
// `abort`, marks every sequence's status RF_ERR_TIMEOUT and returns false; waiters
// that see `abort` return false.  `n` counts this CTA's barriers (thread 0).
static __device__ bool grid_barrier(const BatchParams &P, unsigned int &n)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        GridSync *gs = P.gs;
        int ok = 1;
        volatile int *vabort = &gs->abort;
        if (*vabort) {
            ok = 0;
        } else if (gs->skip && blockIdx.x == 0) {
            ok = 0;  // leave without arriving
        } else {
            const unsigned int target = ++n * gridDim.x;
            // release: the CTA's writes, ordered before thread 0 by __syncthreads, are
            // visible to whoever acquires a later value of count
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&gs->count) : "memory");
            // relaxed polls and one fence at the end: an acquire load drops the SM's L1, which
            // the other CTA may still be scoring from
            long long t0 = 0;
            for (unsigned int polls = 0;; ++polls) {
                unsigned int c;
                asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(&gs->count) : "memory");
                if (c >= target)
                    break;
                if ((polls & 15u) != 0u)
                    continue;
                if (polls == 0)
                    t0 = global_ns();
                if (*vabort) {
                    ok = 0;
                    break;
                }
                if (global_ns() - t0 > P.timeout_ns) {
                    atomicExch(&gs->abort, 1);
                    for (int p = 0; p < P.B; ++p)
                        atomicCAS(P.prob[p].status, 0, RF_ERR_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Block-wide exclusive scan of 0/1 flags; returns this thread's prefix and the total.
__device__ __forceinline__ int block_scan_flag(int flag, int *warp_tot, int *total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const unsigned b = __ballot_sync(0xffffffffu, flag);
    const int in_warp = __popc(b & ((1u << lane) - 1u));
    if (lane == 0)
        warp_tot[w] = __popc(b);
    __syncthreads();
    int before = 0, tot = 0;
    for (int k = 0; k < nw; ++k) {
        if (k < w)
            before += warp_tot[k];
        tot += warp_tot[k];
    }
    __syncthreads();
    *total = tot;
    return before + in_warp;
}

// Merge (max, argmax, second) with another triple; the lowest index wins ties.
__device__ __forceinline__ void merge_max(float &rm, int &am, float &rs, float om, int oa, float os)
{
    float n2 = fmaxf(rs, os);
    if (om > rm || (om == rm && oa >= 0 && (am < 0 || oa < am))) {
        n2 = fmaxf(n2, rm);
        rm = om;
        am = oa;
    } else {
        n2 = fmaxf(n2, om);
    }
    rs = n2;
}

// Sums of eight values over a warp: lane l < 8 returns the total of v[l].  Halving
// the values with every exchange takes 9 FP64 additions where eight butterflies
// take 40 (an FP64 instruction of a warp holds the SM's FP64 unit for 16 clocks).
__device__ __forceinline__ double warp_sum8(double v[8], int lane)
{
#pragma unroll
    for (int h = 4, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return __shfl_sync(0xffffffffu, v[0], ((lane & 4) << 2) | ((lane & 2) << 2) | ((lane & 1) << 2));
}

// Scoring order.  A warp scores particles that are neighbours in the swarm, so
// that its lanes look up neighbouring cells.  The swarm is an anisotropic ball;
// splitting the axis of the largest remaining extent in two, SORT_BITS times,
// gives buckets of about equal sides.  20,000 particles of random order cost 4 to 16 %
// more per lookup.  The order is a stable counting sort, buckets first and particle
// indices inside a bucket, so it is a function of the swarm alone and every sum that
// follows it is the same in every run and for every grid.
// split[s] = axis | depth << 8.
__device__ __forceinline__ void sort_splits(const float r[6], int split[SORT_BITS])
{
    float e[6];
    int depth[6];
    for (int d = 0; d < 6; ++d) {
        e[d] = (d < 3 ? 4.f : 1.f) * r[d];  // a rotation offset moves a point 2 m away by about 4 m per unit
        depth[d] = 0;
    }
    for (int s = 0; s < SORT_BITS; ++s) {
        int a = 0;
        for (int d = 1; d < 6; ++d)
            if (e[d] > e[a])
                a = d;
        split[s] = a | (++depth[a] << 8);
        e[a] *= 0.5f;
    }
}

__device__ __forceinline__ int sort_key(const float *pst, int ld, int i, const int split[SORT_BITS])
{
    int key = 0;
#pragma unroll
    for (int s = 0; s < SORT_BITS; ++s) {
        const int a = split[s] & 255, depth = split[s] >> 8;
        // a coordinate of the uniform 6-ball lies in [-0.7, 0.7] for 97 % of the particles
        const float x = __saturatef(fmaf(__ldg(&pst[(size_t)a * ld + i]), 0.7f, 0.5f));
        const int q = min((int)(x * (float)(1 << depth)), (1 << depth) - 1);
        key = 2 * key + (q & 1);
    }
    return key;
}

// First pass of the sort, one block of SORT_BLOCK particles by one CTA: every particle's
// bucket, its place among the block's earlier particles of that bucket, and the block's
// counts.  A warp takes consecutive particles, 32 at a time, and counts them in its own
// row of `rows` (FIT_WARPS x SORT_BUCKETS, shared memory); the particles of a round that
// share a bucket find each other by __match_any_sync, so no place depends on the order of
// arrival.
// Bound by latency: loads, SORT_ROUNDS dependent rounds and the prefix.  Blocks of 512
// particles, ranked beside the point tests by CTAs that take no points: 10,000 / 20,000
// particle frames 2519 / 14275 us; blocks of 1024 2541 / 14423, of 256 2519 / 14311.  Global
// counters with atomic arrival order took 2533 / 14407 us and ranked a bucket's particles
// differently in every run.
constexpr int SORT_ROUNDS = SORT_BLOCK / FIT_THREADS;
static __device__ void sort_count(const ProblemDesc &pd, int n, int blk, const int split[SORT_BITS], uint16_t *rows)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    __syncthreads();
    for (int q = tid; q < FIT_WARPS * SORT_BUCKETS / 8; q += FIT_THREADS)
        reinterpret_cast<uint4 *>(rows)[q] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    uint16_t *row = rows + w * SORT_BUCKETS;
    const int i0 = blk * SORT_BLOCK + w * (SORT_BLOCK / FIT_WARPS) + lane;
    int key[SORT_ROUNDS], place[SORT_ROUNDS];
#pragma unroll
    for (int r = 0; r < SORT_ROUNDS; ++r)
        key[r] = i0 + 32 * r < n ? sort_key(pd.pst, pd.n_tmpl, i0 + 32 * r, split) : -1;
#pragma unroll
    for (int r = 0; r < SORT_ROUNDS; ++r) {
        const unsigned same = __match_any_sync(0xffffffffu, key[r]);
        const unsigned before = same & ((1u << lane) - 1u);
        const int old = key[r] >= 0 ? row[key[r]] : 0;
        place[r] = old + __popc(before);
        __syncwarp();
        if (key[r] >= 0 && before == 0u)
            row[key[r]] = (uint16_t)(old + __popc(same));
        __syncwarp();
    }
    __syncthreads();
    // four buckets a thread: a warp's row becomes the counts of the warps before it
    unsigned c[4] = {0u, 0u, 0u, 0u};
    for (int q = 0; q < FIT_WARPS; ++q) {
        uint2 *at = reinterpret_cast<uint2 *>(rows + q * SORT_BUCKETS) + tid;
        const uint2 v = *at;
        *at = make_uint2(c[0] | c[1] << 16, c[2] | c[3] << 16);
        c[0] += v.x & 0xFFFFu;
        c[1] += v.x >> 16;
        c[2] += v.y & 0xFFFFu;
        c[3] += v.y >> 16;
    }
    reinterpret_cast<uint2 *>(pd.bucket_counts + (size_t)blk * SORT_BUCKETS)[tid] =
        make_uint2(c[0] | c[1] << 16, c[2] | c[3] << 16);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < SORT_ROUNDS; ++r)
        if (key[r] >= 0)
            pd.key[i0 + 32 * r] = key[r] | (place[r] + row[key[r]]) << SORT_BITS;
}

// Second pass, after a grid barrier: the same block's particles to their places, which
// follow the smaller buckets, then the bucket's particles of the blocks before.
// `at` holds SORT_BUCKETS + FIT_WARPS ints of shared memory.
static __device__ void sort_place(const ProblemDesc &pd, int n, int blk, int *at)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int n_blocks = (n + SORT_BLOCK - 1) / SORT_BLOCK;
    const int i0 = blk * SORT_BLOCK + tid;
    int kp[SORT_ROUNDS];
#pragma unroll
    for (int r = 0; r < SORT_ROUNDS; ++r)
        kp[r] = i0 + FIT_THREADS * r < n ? __ldcg(&pd.key[i0 + FIT_THREADS * r]) : 0;
    int all[4] = {0, 0, 0, 0}, before[4] = {0, 0, 0, 0};
#pragma unroll 8
    for (int q = 0; q < n_blocks; ++q) {
        const uint2 v = __ldcg(reinterpret_cast<const uint2 *>(pd.bucket_counts + (size_t)q * SORT_BUCKETS) + tid);
        const int c[4] = {(int)(v.x & 0xFFFFu), (int)(v.x >> 16), (int)(v.y & 0xFFFFu), (int)(v.y >> 16)};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            all[e] += c[e];
            before[e] += q < blk ? c[e] : 0;
        }
    }
    const int mine = all[0] + all[1] + all[2] + all[3];
    int inc = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, inc, o);
        inc += lane >= o ? up : 0;
    }
    int *warp_sum = at + SORT_BUCKETS;
    __syncthreads();
    if (lane == 31)
        warp_sum[w] = inc;
    __syncthreads();
    int first = inc - mine;
    for (int q = 0; q < w; ++q)
        first += warp_sum[q];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        at[4 * tid + e] = first + before[e];
        first += all[e];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < SORT_ROUNDS; ++r) {
        const int i = i0 + FIT_THREADS * r;
        if (i < n) {
            const int slot = at[kp[r] & (SORT_BUCKETS - 1)] + (kp[r] >> SORT_BITS);
            pd.ord[slot] = i;
            if (i == 0)
                pd.ord[pd.n_tmpl] = slot;
        }
    }
}

// Per-sequence state, identical in every CTA (computed redundantly in a fixed order).
struct PState {
    Pose c, prev;
    float r[6], r1[6];
    float rho_carry, rho_ref;
    int empty_run, stop, active, iters;
    int level, n_lvl, m_lvl, off_lvl;
    int nO, offset;
    int groups, n_chunks, chunk, unit_base;
    int sorted, split[SORT_BITS];
    long long lookups;
};

// ------------------------------------------------------------------ the persistent kernel
template <int DT, int MODE, int LG>
__global__ void __launch_bounds__(FIT_THREADS, RF_PFO_MIN_BLOCKS) pfo_batch_kernel(const __grid_constant__ BatchParams P)
{
    extern __shared__ ulonglong2 smem_raw[];
    __shared__ PState st[MAX_BATCH];
    __shared__ int warp_tot[FIT_WARPS];
    __shared__ double share_S[FIT_WARPS][32];
    __shared__ int share_n[FIT_WARPS][32];
    __shared__ double red_d[FIT_WARPS];
    __shared__ float red_f[2];
    __shared__ int red_i[3];
    static_assert(FIT_WARPS == 8, "phase C: one warp per APS quantity");
    __shared__ int s_total_units;
    static_assert(SORT_BUCKETS == 4 * FIT_THREADS, "four buckets per thread");
    static_assert(SORT_BLOCK == SORT_ROUNDS * FIT_THREADS, "whole rounds of a block");
    static_assert(FIT_WARPS * SORT_BUCKETS * sizeof(uint16_t) <= FIT_WARPS * sizeof(PairPoints) &&
                      (SORT_BUCKETS + FIT_WARPS) * sizeof(int) <= FIT_WARPS * sizeof(PairPoints),
                  "the sort works in the points' shared memory");

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int G = gridDim.x, b = blockIdx.x;
    const int B = P.B;
    unsigned int n_barriers = 0;

    // ---- prologue: clear the statistics and statuses (here and not by one memset each:
    // a stream operation costs a small frame about 2 us), unproject the points of every
    // level of every sequence (Eq. unproj)
    for (int p = b; p < B; p += G) {
        if (P.prob[p].stats)
            for (int i = tid; i < (int)(sizeof(rf_frame_stats) / sizeof(int)); i += blockDim.x)
                reinterpret_cast<int *>(P.prob[p].stats)[i] = 0;
        if (tid == 0)
            *P.prob[p].status = 0;
    }
    {
        long long total = 0;
        for (int p = 0; p < B; ++p)
            total += P.prob[p].m_all;
        for (long long g = (long long)b * blockDim.x + tid; g < total; g += (long long)G * blockDim.x) {
            int p = 0;
            long long base = 0;
            while (g >= base + P.prob[p].m_all) {
                base += P.prob[p].m_all;
                ++p;
            }
            const ProblemDesc &pd = P.prob[p];
            const int j = (int)(g - base);
            int l = 0;
            while (l + 1 < pd.n_levels && j >= pd.lvl_off[l + 1])
                ++l;
            float4 pt;
            unproject_point(pd.depth, pd.K, pd.lvl_stride[l], pd.lvl_nw[l], j - pd.lvl_off[l], pt);
            pd.pts[j] = pt;
        }
    }
    if (tid < B) {
        const ProblemDesc &pd = P.prob[tid];
        PState &s = st[tid];
        const float *c0 = pd.init_pose ? pd.init_pose : pd.prev_pose;
        for (int a = 0; a < 4; ++a) {
            s.c.q[a] = __ldcg(&c0[a]);
            s.prev.q[a] = __ldcg(&pd.prev_pose[a]);
        }
        for (int a = 0; a < 3; ++a) {
            s.c.t[a] = __ldcg(&c0[4 + a]);
            s.prev.t[a] = __ldcg(&pd.prev_pose[4 + a]);
        }
        for (int d = 0; d < 6; ++d)
            s.r[d] = s.r1[d] = __ldcg(&pd.scale[d]);
        s.rho_carry = 0.f;
        s.rho_ref = 0.f;
        s.empty_run = 0;
        // stop code 5: skipped by the caller's run flag (never active, writes nothing)
        s.stop = (pd.run_flag && __ldcg(pd.run_flag) == 0) ? 5 : 0;
        s.iters = 0;
        s.lookups = 0;
    }
    if (!grid_barrier(P, n_barriers))
        return;

    for (int k = 1; k <= P.k_max_all; ++k) {
        if (tid < B) {
            const ProblemDesc &pd = P.prob[tid];
            PState &s = st[tid];
            s.active = (s.stop == 0 && k <= pd.k_max) ? 1 : 0;
            const int l = (k - 1) % pd.n_levels;
            s.level = l;
            s.n_lvl = pd.lvl_n[l];
            s.m_lvl = pd.lvl_m[l];
            s.off_lvl = pd.lvl_off[l];
            s.sorted = s.active && (long long)s.n_lvl * s.m_lvl >= SORT_MIN_WORK;
            if (s.active)
                s.iters = k;
            if (s.sorted)
                sort_splits(s.r, s.split);
        }
        __syncthreads();
        int T = 0, sort_blocks = 0;
        bool any = false;
        for (int p = 0; p < B; ++p)
            if (st[p].active) {
                any = true;
                T += st[p].m_lvl;
                sort_blocks += st[p].sorted ? (st[p].n_lvl + SORT_BLOCK - 1) / SORT_BLOCK : 0;
            }
        if (!any)
            break;  // identical decision in every CTA
        // The last CTAs order the swarms, one block of particles each, while the others take the
        // points: neither waits for the other.
        const int n_sort = min(sort_blocks, G / 2);
        auto each_block = [&](auto &&f) {
            if (b < G - n_sort)
                return;
            for (int q = G - 1 - b; q < sort_blocks; q += n_sort) {
                int p = 0, blk = q;
                for (;; ++p) {
                    const int n = st[p].sorted ? (st[p].n_lvl + SORT_BLOCK - 1) / SORT_BLOCK : 0;
                    if (blk < n)
                        break;
                    blk -= n;
                }
                if (st[p].active)
                    f(P.prob[p], st[p], blk);
            }
        };
        // ---- phase A: overlap counts per (CTA, sequence) over the concatenated point sets
        const int seg = (T + G - n_sort - 1) / (G - n_sort);
        const int jb = min(T, b * seg), je = min(T, jb + seg);
        {
            int base = 0;
            for (int p = 0; p < B; ++p) {
                if (!st[p].active)
                    continue;
                const ProblemDesc &pd = P.prob[p];
                const int lo = max(jb, base), hi = min(je, base + st[p].m_lvl);
                int cnt = 0;
                if (lo < hi) {
                    float Rc[9], Rp[9];
                    quat_rot(st[p].c.q, Rc);
                    quat_rot(st[p].prev.q, Rp);
                    const bool overlap_on = (pd.flags & RF_OVERLAP) != 0;
                    const float cell_m = (pd.flags & RF_CELL_MARGIN) ? 1.7320508f * pd.V.voxel : 0.f;
                    for (int j0 = lo; j0 < hi; j0 += blockDim.x) {
                        const int j = j0 + tid;
                        int f = 0;
                        if (j < hi) {
                            const float4 pt = __ldcg(&pd.pts[st[p].off_lvl + (j - base)]);
                            f = overlap_on ? overlap_test(pt, Rc, st[p].c.t, Rp, st[p].prev.t, pd.prev_depth, pd.K, cell_m)
                                           : (pt.w != 0.f);
                        }
                        int tot;
                        block_scan_flag(f, warp_tot, &tot);
                        cnt += tot;
                    }
                }
                if (tid == 0)
                    P.block_counts[(size_t)b * MAX_BATCH + p] = cnt;
                base += st[p].m_lvl;
            }
        }
        each_block([&](const ProblemDesc &pd, const PState &s, int blk) {
            sort_count(pd, s.n_lvl, blk, s.split, reinterpret_cast<uint16_t *>(smem_raw));
        });
        if (!grid_barrier(P, n_barriers))
            return;
        // ---- phase A': per-sequence offsets and |O_k|, then the compaction
        for (int p = w; p < B; p += FIT_WARPS) {
            if (!st[p].active)
                continue;
            int before = 0, tot = 0;
            for (int q = lane; q < G; q += 32) {
                const int c = __ldcg(&P.block_counts[(size_t)q * MAX_BATCH + p]);
                tot += c;
                before += (q < b) ? c : 0;
            }
            for (int o = 16; o > 0; o >>= 1) {
                tot += __shfl_xor_sync(0xffffffffu, tot, o);
                before += __shfl_xor_sync(0xffffffffu, before, o);
            }
            if (lane == 0) {
                st[p].nO = tot;
                st[p].offset = before;
            }
        }
        __syncthreads();
        if (tid < B && st[tid].active && st[tid].nO == 0) {  // empty overlap: this sequence stops
            PState &s = st[tid];
            s.stop = 4;
            s.active = 0;
            if (b == 0) {
                atomicCAS(P.prob[tid].status, 0, RF_ERR_EMPTY);
                if (P.prob[tid].stats) {
                    rf_iter_stats &row = P.prob[tid].stats->it[k - 1];
                    memset(&row, 0, sizeof row);
                    row.k = k;
                    row.stop = 4;
                    row.level = s.level;
                    row.n_particles = s.n_lvl;
                }
            }
        }
        __syncthreads();
        {
            int base = 0;
            for (int p = 0; p < B; ++p) {
                if (!(st[p].active || (st[p].stop == 4 && st[p].nO == 0 && st[p].iters == k)))
                    continue;  // only sequences that took part in phase A (their points count in T)
                const ProblemDesc &pd = P.prob[p];
                const int lo = max(jb, base), hi = min(je, base + st[p].m_lvl);
                if (lo < hi && st[p].active) {
                    float Rc[9], Rp[9];
                    quat_rot(st[p].c.q, Rc);
                    quat_rot(st[p].prev.q, Rp);
                    const bool overlap_on = (pd.flags & RF_OVERLAP) != 0;
                    const float cell_m = (pd.flags & RF_CELL_MARGIN) ? 1.7320508f * pd.V.voxel : 0.f;
                    int out = st[p].offset;
                    for (int j0 = lo; j0 < hi; j0 += blockDim.x) {
                        const int j = j0 + tid;
                        int f = 0;
                        float4 pt = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (j < hi) {
                            pt = __ldcg(&pd.pts[st[p].off_lvl + (j - base)]);
                            f = overlap_on ? overlap_test(pt, Rc, st[p].c.t, Rp, st[p].prev.t, pd.prev_depth, pd.K, cell_m)
                                           : (pt.w != 0.f);
                        }
                        int tot;
                        const int pos = block_scan_flag(f, warp_tot, &tot);
                        if (f)
                            pd.cpts[out + pos] = pt;
                        out += tot;
                    }
                }
                base += st[p].m_lvl;
            }
        }
        each_block([&](const ProblemDesc &pd, const PState &s, int blk) {
            sort_place(pd, s.n_lvl, blk, reinterpret_cast<int *>(smem_raw));
        });
        if (!grid_barrier(P, n_barriers))
            return;
        // ---- phase B: fitness of every particle of every active sequence (Eq. normallh)
        if (tid == 0) {
            int units = 0;
            for (int p = 0; p < B; ++p) {
                PState &s = st[p];
                if (!s.active)
                    continue;
                const Split sp = make_split(s.n_lvl, s.nO, P.work_warps, P.prob[p].max_chunks);
                s.groups = sp.groups;
                s.n_chunks = sp.n_chunks;
                s.chunk = sp.chunk;
                s.unit_base = units;
                units += sp.groups * sp.n_chunks;
            }
            s_total_units = units;
        }
        __syncthreads();
        {
            const int total_units = s_total_units;
            PairPoints &spts = reinterpret_cast<PairPoints *>(smem_raw)[w];
            int *ctr = P.unit_ctr + (k - 1);
            int t = 0;
            if (lane == 0)
                t = atomicAdd(ctr, 1);
            int u = __shfl_sync(0xffffffffu, t, 0);
            while (u < total_units) {
                if (lane == 0)
                    t = atomicAdd(ctr, 1);
                const int u_next = __shfl_sync(0xffffffffu, t, 0);
                // the last active sequence whose first unit is <= u (active bases increase)
                int p = 0;
                for (int q = 0; q < B; ++q)
                    if (st[q].active && st[q].unit_base <= u)
                        p = q;
                const PState &s = st[p];
                const ProblemDesc &pd = P.prob[p];
                const int local = u - s.unit_base;
                const int ch = local / s.groups, g = local - ch * s.groups;
                const int j0 = ch * s.chunk;
                const int cnt = min(s.chunk, s.nO - j0);
                __syncwarp();
                for (int j = lane; j < cnt; j += 32)
                    stage_point(spts, j, __ldcg(&pd.cpts[j0 + j]));
                __syncwarp();
                FitParams fp;
                fp.pst = pd.pst;
                fp.n = s.n_lvl;
                fp.ld = pd.n_tmpl;
                fp.c = s.c;
                for (int d = 0; d < 6; ++d)
                    fp.r[d] = s.r[d];
                fp.l1 = (pd.flags & RF_L1) != 0;
                fp.right_mult = (pd.flags & RF_RIGHT_MULT) != 0;
                // a lane's two particles are 32 places apart in the scoring order
                const int slot[2] = {g * GROUP_PARTICLES + lane, g * GROUP_PARTICLES + 32 + lane};
                int i[2], nv[2];
                double S[2];
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    i[h] = slot[h] < s.n_lvl && s.sorted ? __ldcg(&pd.ord[slot[h]]) : slot[h];
                fitness_unit<DT, MODE, LG>(pd.V, spts, cnt, fp, i, S, nv);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (slot[h] < s.n_lvl) {  // stored [chunk][place]: a warp's partials are contiguous
                        pd.part_S[(size_t)ch * s.n_lvl + slot[h]] = S[h];
                        pd.part_n[(size_t)ch * s.n_lvl + slot[h]] = nv[h];
                    }
                u = u_next;
            }
        }
        if (!grid_barrier(P, n_barriers))
            return;
        // ---- phase B': per-particle totals, rho, per-CTA APS sums (Eq. ebs, Eq. wafit)
        for (int p = 0; p < B; ++p) {
            if (!st[p].active)
                continue;
            const ProblemDesc &pd = P.prob[p];
            const bool normalize = (pd.flags & RF_NORMALIZE) != 0;
            // A warp's lanes are 32 neighbours of the scoring order and its chunks every FIT_WARPS-th,
            // so every load of a partial is a contiguous run; the warps' sums meet in shared
            // memory in a fixed order.  CTA b takes places 32 b .. 32 b + 31, 32 (b + G) ..
            // Bound by the FP64 additions (one a partial).  A warp per particle with its lanes
            // over the chunks needs as many again for the butterfly: 37 us an iteration at
            // 20,000 particles x 94 chunks against 13, 15 against 6 at 1024 x 110.
            const int n_lvl = st[p].n_lvl, n_chunks = st[p].n_chunks;
            auto share = [&](int slot) {
                double S = 0.0;
                int nv = 0;
                if (slot < n_lvl) {
#pragma unroll 8
                    for (int ch = w; ch < n_chunks; ch += FIT_WARPS) {
                        S += __ldcg(&pd.part_S[(size_t)ch * n_lvl + slot]);
                        nv += __ldcg(&pd.part_n[(size_t)ch * n_lvl + slot]);
                    }
                }
                share_S[w][lane] = S;
                share_n[w][lane] = nv;
            };
            auto total = [&](int l, double &S, int &nv) {
                S = share_S[0][l];
                nv = share_n[0][l];
#pragma unroll
                for (int q = 1; q < FIT_WARPS; ++q) {
                    S += share_S[q][l];
                    nv += share_n[q][l];
                }
            };
            const bool centre = k == 1 || (pd.flags & RF_RHO_REF_CENTER) || pd.n_levels > 1;
            if (centre) {  // the centre particle's total, by the same sums as every particle's below
                share(lane != 0 ? n_lvl : (st[p].sorted ? __ldcg(&pd.ord[pd.n_tmpl]) : 0));
                __syncthreads();
            }
            if (tid == 0) {
                double S0 = 0.0;
                int n0;
                if (centre)
                    total(0, S0, n0);
                st[p].rho_ref = centre ? fitness_rho(S0, st[p].nO, pd.tau, normalize) : st[p].rho_carry;
            }
            __syncthreads();
            if (b * 32 >= n_lvl)
                continue;  // no particles of this sequence for the CTA
            const float rho_ref = st[p].rho_ref;
            // particle 0 is the centre s*_{k-1} itself: an APS candidate only with RF_APS_WITH_CENTRE
            const int first = (pd.flags & RF_APS_WITH_CENTRE) ? 0 : 1;
            double sw = 0.0, swr = 0.0, swd[6] = {0, 0, 0, 0, 0, 0};
            int naps = 0, amax = -1;
            int valid = 0;  // whether any particle has a valid TSDF sample (first corner case of Sec. 4)
            float rmax = -1.f, r2 = -1.f;
            for (int i0 = b * 32; i0 < n_lvl; i0 += G * 32) {
                share(i0 + lane);
                __syncthreads();
                if (w == 0 && i0 + lane < n_lvl) {
                    const int i = st[p].sorted ? __ldcg(&pd.ord[i0 + lane]) : i0 + lane;
                    double S;
                    int nv;
                    total(lane, S, nv);
                    valid |= nv != 0;
                    const float rho = fitness_rho(S, st[p].nO, pd.tau, normalize);
                    merge_max(rmax, amax, r2, rho, i, -1.f);
                    if (i >= first && rho > rho_ref) {
                        const double wgt = (double)(rho - rho_ref);
                        ++naps;
                        sw += wgt;
                        swr += wgt * (double)rho;
#pragma unroll
                        for (int d = 0; d < 6; ++d)
                            swd[d] += wgt * (double)(st[p].r[d] * __ldg(&pd.pst[(size_t)d * pd.n_tmpl + i]));
                    }
                }
                __syncthreads();
            }
            if (w == 0) {  // the CTA's sums
                double acc[8] = {sw, swr, swd[0], swd[1], swd[2], swd[3], swd[4], swd[5]};
                const double mine = warp_sum8(acc, lane);
                valid = __any_sync(0xffffffffu, valid);
                for (int o = 16; o > 0; o >>= 1) {
                    const float om = __shfl_xor_sync(0xffffffffu, rmax, o);
                    const int oa = __shfl_xor_sync(0xffffffffu, amax, o);
                    const float o2 = __shfl_xor_sync(0xffffffffu, r2, o);
                    merge_max(rmax, amax, r2, om, oa, o2);
                }
                naps = __reduce_add_sync(0xffffffffu, naps);
                double *out = P.aps + ((size_t)b * MAX_BATCH + p) * APW;
                if (lane < 8)
                    out[lane] = mine;
                if (lane == 8)  // |APS| with a sign bit for "some valid sample", max, argmax, second
                    *reinterpret_cast<int4 *>(out + 8) = make_int4(naps | (valid ? (int)0x80000000 : 0), __float_as_int(rmax),
                                                                   amax, __float_as_int(r2));
            }
        }
        if (!grid_barrier(P, n_barriers))
            return;
        // ---- phase C: fixed-order reduction of the APS sums and the PST update, the same in
        // every CTA.  Warp e sums the CTAs' partials of quantity e (15 FP64 additions a warp;
        // an FP64 instruction holds the SM's unit for 16 clocks, and both its CTAs do this);
        // the last warp also merges the maxima and counts.  Then warp 0 updates the sequence
        // with one axis per lane, so that the FP64 divisions of the six axes run side by side
        // instead of one after another.  (One warp for everything took 17 to 20 us an
        // iteration; this takes 5 at 1024 particles, 10 at 20,000.)
        for (int p = 0; p < B; ++p) {
            if (!st[p].active)
                continue;
            const int parts = min(G, (st[p].n_lvl + 31) / 32);  // CTAs that had particles
            {
                double acc = 0.0;
                for (int q = lane; q < parts; q += 32)
                    acc += __ldcg(&P.aps[((size_t)q * MAX_BATCH + p) * APW + w]);
                for (int o = 16; o > 0; o >>= 1)
                    acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0)
                    red_d[w] = acc;
                if (w == FIT_WARPS - 1) {
                    int na = 0, am = -1, any = 0;
                    float rm = -1.f, rs = -1.f;
                    for (int q = lane; q < parts; q += 32) {
                        const int4 v = __ldcg(reinterpret_cast<const int4 *>(P.aps + ((size_t)q * MAX_BATCH + p) * APW + 8));
                        na += v.x & 0x7FFFFFFF;
                        any |= v.x < 0;
                        merge_max(rm, am, rs, __int_as_float(v.y), v.z, __int_as_float(v.w));
                    }
                    for (int o = 16; o > 0; o >>= 1) {
                        const float om = __shfl_xor_sync(0xffffffffu, rm, o);
                        const int oa = __shfl_xor_sync(0xffffffffu, am, o);
                        const float o2 = __shfl_xor_sync(0xffffffffu, rs, o);
                        merge_max(rm, am, rs, om, oa, o2);
                    }
                    na = __reduce_add_sync(0xffffffffu, na);
                    any = __any_sync(0xffffffffu, any);
                    if (lane == 0) {
                        red_f[0] = rm;
                        red_f[1] = rs;
                        red_i[0] = am;
                        red_i[1] = na;
                        red_i[2] = any;
                    }
                }
            }
            __syncthreads();
            if (w == 0) {
                const double v = lane < 8 ? red_d[lane] : 0.0;
                const float rm = red_f[0], rs = red_f[1];
                const int am = red_i[0], na = red_i[1];
                const ProblemDesc &pd = P.prob[p];
                PState &s = st[p];
                // first corner case of Sec. 4: no particle found a single TSDF sample, so the
                // likelihood cannot be evaluated: rho = 0.5, v = 1, r_hat = 0.5 v + eps, s* kept
                const int corner = red_i[2] == 0 ? 1 : (na == 0 ? 2 : 0);
                const int n_aps = corner == 1 ? 0 : na;
                const float rho_ref = s.rho_ref;
                // lane 1: Eq. wafit; lanes 2 .. 7: the offsets of Eq. ebs, axis d on lane 2 + d
                const double sw = __shfl_sync(0xffffffffu, v, 0);
                const double quo = n_aps > 0 ? v / sw : 0.0;
                const float rho_t = corner == 1 ? 0.5f : (n_aps > 0 ? (float)__shfl_sync(0xffffffffu, quo, 1) : rho_ref);
                float dbar[6];
                double nv2 = 0.0;
#pragma unroll
                for (int d = 0; d < 6; ++d) {
                    const double db = __shfl_sync(0xffffffffu, quo, 2 + d);
                    dbar[d] = (float)db;
                    nv2 += db * db;
                }
                const double nv = sqrt(nv2);
                float rhat;
                if (corner == 1) {
                    rhat = (float)(0.5 + (double)pd.eps);
                } else if (n_aps > 0) {
                    const double dir = nv < 1e-12 ? 0.40824829046386302 : fabs(quo) / nv;
                    rhat = (float)((1.0 - (double)rho_t) * dir + (double)pd.eps);
                } else {
                    rhat = (float)(2.0 * (1.0 - (double)rho_ref) * 0.40824829046386302 + (double)pd.eps);
                }
                if (lane >= 2 && lane < 8) {
                    const int d = lane - 2;
                    s.r[d] = pd.beta * s.r[d] + (1.f - pd.beta) * rhat;
                    if (k == 1)
                        s.r1[d] = s.r[d];
                }
                __syncwarp();
                if (lane == 0) {
                    if (n_aps > 0) {
                        Pose s_new;
                        compose_offset(s.c, dbar, (pd.flags & RF_RIGHT_MULT) != 0, s_new);
                        s.c = s_new;
                        s.empty_run = 0;
                    } else {
                        s.empty_run += 1;
                    }
                    s.rho_carry = rho_t;
                    float step = 0.f;
                    for (int d = 0; d < 6; ++d)
                        step = fmaxf(step, fabsf(dbar[d]));
                    int stop = 0;
                    if (s.empty_run >= 2)
                        stop = 1;
                    else if (n_aps > 0 && step < pd.stop_eps)
                        stop = 2;
                    else if (k == pd.k_max)
                        stop = 3;
                    s.stop = stop;
                    s.lookups += (long long)s.nO * (long long)s.n_lvl;
                    if (b == 0 && pd.stats) {
                        rf_iter_stats &row = pd.stats->it[k - 1];
                        row.k = k;
                        row.n_overlap = s.nO;
                        row.n_aps = n_aps;
                        row.argmax = am;
                        row.rho_ref = rho_ref;
                        row.rho_tilde = rho_t;
                        row.rho_max = rm;
                        row.rho_second = rs;
                        for (int a = 0; a < 4; ++a)
                            row.pose[a] = s.c.q[a];
                        for (int a = 0; a < 3; ++a)
                            row.pose[4 + a] = s.c.t[a];
                        for (int d = 0; d < 6; ++d) {
                            row.scale[d] = s.r[d];
                            row.offset[d] = dbar[d];
                        }
                        row.stop = stop;
                        row.level = s.level;
                        row.n_particles = s.n_lvl;
                        row.corner = corner;
                    }
                }
            }
            __syncthreads();
        }
    }
    // ---- epilogue (CTA 0): final poses, r_1 for the next frame, summaries
    if (b == 0 && tid < B && st[tid].stop != 5) {
        const ProblemDesc &pd = P.prob[tid];
        const PState &s = st[tid];
        for (int a = 0; a < 4; ++a)
            pd.out_pose[a] = s.c.q[a];
        for (int a = 0; a < 3; ++a)
            pd.out_pose[4 + a] = s.c.t[a];
        for (int d = 0; d < 6; ++d)
            pd.scale[d] = s.r1[d];
        if (pd.stats) {
            pd.stats->iters = s.iters;
            pd.stats->status = *((volatile int *)pd.status);
            pd.stats->n_points = pd.lvl_m[0];
            pd.stats->lookups = s.lookups;
            for (int d = 0; d < 6; ++d)
                pd.stats->r1[d] = s.r1[d];
        }
    }
}

// ------------------------------------------------------------------ kernel table
// The trilinear modes are built for groups of 4, 6 and 8 lookups in flight (the
// group regroups the FP32 partial sums, so results differ in rounding only);
// nearest-voxel modes sample one point at a time and have one variant.  Each
// storage type's variants live in their own translation unit.
using PfoFn = void (*)(BatchParams);
constexpr int GROUP_CHOICES[3] = {4, 6, 8};
template <int DT, int MODE> PfoFn pfo_fn_group(int group)
{
    if constexpr ((MODE & 1) != 0) {
        return pfo_batch_kernel<DT, MODE, GROUP>;
    } else {
        switch (group) {
        case 4:
            return pfo_batch_kernel<DT, MODE, 4>;
        case 8:
            return pfo_batch_kernel<DT, MODE, 8>;
        default:
            return pfo_batch_kernel<DT, MODE, GROUP>;
        }
    }
}
template <int DT> PfoFn pfo_fn_dtype(int mode, int group)
{
    switch (mode) {
    case 0:
        return pfo_fn_group<DT, 0>(group);
    case 1:
        return pfo_fn_group<DT, 1>(group);
    case 2:
        return pfo_fn_group<DT, 2>(group);
    default:
        return pfo_fn_group<DT, 3>(group);
    }
}
PfoFn pfo_fn_f32(int mode, int group);
PfoFn pfo_fn_f16(int mode, int group);
PfoFn pfo_fn_i16(int mode, int group);

}  // namespace rf
