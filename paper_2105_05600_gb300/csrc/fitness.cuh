// fitness.cuh -- device code shared by the standalone fitness kernels (track.cu)
// and the persistent PFO kernel (pfo.cu): point unprojection, the overlap test of
// Eq. validness, the warp-level fitness of Eq. normallh over packed TSDF cells, the
// work split into (particle group, point chunk) units and the per-particle totals.
#pragma once

#include <algorithm>

#include "common.cuh"

namespace rf {


Pose to_pose(const rf_pose &p);

constexpr int FIT_THREADS = 256;
constexpr int FIT_WARPS = FIT_THREADS / 32;
constexpr int GROUP_PARTICLES = 64;   // particles of a warp's work unit, two per lane
constexpr int CHUNK_MAX = 256;        // points staged at once
constexpr int MIN_CHUNK = 32;         // fewest points per work unit
constexpr int SMALL_CHUNK = 24;       // fewest where there are not enough units for the warps
#ifndef RF_UNITS_PER_WARP
#define RF_UNITS_PER_WARP 16
#endif
constexpr int UNITS_PER_WARP = RF_UNITS_PER_WARP;  // target work units per warp and iteration
constexpr int APW = 16;               // doubles per CTA in the APS partials: 8 sums, then one int4
constexpr int MAX_CTAS_PER_SM = 2048 / FIT_THREADS;  // bound for grid-sized scratch
// CTAs of the persistent kernel resident per SM (register budget 65536 / (256 * n)).
// 3 leave 80 registers for the pair loop, which spills: 15.7 ms against 13.9 ms for a
// paper-scale frame.
#ifndef RF_PFO_MIN_BLOCKS
#define RF_PFO_MIN_BLOCKS 2
#endif
// Points whose terms are added before the compensated sum, half of them (for two
// particles each: GROUP lookups) with their loads in flight together; the default.
// The persistent kernel is also built for 4 and 8, picked by the launch configuration.
#ifndef RF_GROUP
#define RF_GROUP 6
#endif
constexpr int GROUP = RF_GROUP;

// ------------------------------------------------------------------ small helpers
__device__ __forceinline__ long long global_ns()
{
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void unproject_point(const float *__restrict__ depth, const Intr &K, int stride, int nw,
                                                int j, float4 &out)
{
    const int a = j % nw, b = j / nw;
    const int u = a * stride, v = b * stride;
    const float z = depth[(size_t)v * K.width + u];
    if (depth_valid(z, K))
        out = make_float4(((float)u - K.cx) * z / K.fx, ((float)v - K.cy) * z / K.fy, z, 1.f);
    else
        out = make_float4(0.f, 0.f, 0.f, 0.f);
}

// Eq. validness for one point: world with the current estimate (Rc, tc), back
// into frame t-1 with its final pose (Rp, tp), nearest pixel, valid depth.
// cell_m > 0 (RF_CELL_MARGIN: sqrt(3) voxels) also keeps the continuous pixel
// position fx cell_m / z' pixels inside the image edges, so that the TSDF cell
// the point samples lies inside frame t-1's view.
__device__ __forceinline__ bool overlap_test(const float4 &p, const float Rc[9], const float tc[3], const float Rp[9],
                                             const float tp[3], const float *__restrict__ prev_depth, const Intr &K,
                                             float cell_m)
{
    if (p.w == 0.f)
        return false;
    const float gx = Rc[0] * p.x + Rc[1] * p.y + Rc[2] * p.z + tc[0] - tp[0];
    const float gy = Rc[3] * p.x + Rc[4] * p.y + Rc[5] * p.z + tc[1] - tp[1];
    const float gz = Rc[6] * p.x + Rc[7] * p.y + Rc[8] * p.z + tc[2] - tp[2];
    const float cx = Rp[0] * gx + Rp[3] * gy + Rp[6] * gz;
    const float cy = Rp[1] * gx + Rp[4] * gy + Rp[7] * gz;
    const float cz = Rp[2] * gx + Rp[5] * gy + Rp[8] * gz;
    if (!(cz > 0.f))
        return false;
    const float uc = K.fx * cx / cz + K.cx, vc = K.fy * cy / cz + K.cy;
    const float mu = K.fx * cell_m / cz, mv = K.fy * cell_m / cz;
    if (!(uc >= mu - 0.5f && uc < (float)K.width - 0.5f - mu && vc >= mv - 0.5f && vc < (float)K.height - 0.5f - mv))
        return false;
    const float u = floorf(uc + 0.5f);
    const float v = floorf(vc + 0.5f);
    if (!(u >= 0.f && u < (float)K.width && v >= 0.f && v < (float)K.height))
        return false;
    const float d = __ldg(&prev_depth[(size_t)v * K.width + (size_t)u]);
    return depth_valid(d, K);
}

// ------------------------------------------------------------------ fitness (warp level)
// MODE bit 0: nearest sample; bit 1: plain (uncompensated) FP32 sum.
template <int MODE> struct Mode {
    static constexpr bool nearest = (MODE & 1) != 0;
    static constexpr bool plain = (MODE & 2) != 0;
};

struct FitParams {
    const float *pst;   // template, structure of arrays with leading dimension ld (pst[d * ld + i])
    int n;              // particles scored: the first n rows of the template
    int ld;
    Pose c;             // PST centre
    float r[6];         // axis lengths
    int l1, right_mult;
};

// Pose of particle i (centre (+) (scale . omega_i)), folded with the world ->
// voxel-centre map g = p / voxel - origin / voxel - 1/2, so that a point goes
// straight to grid units.
__device__ __forceinline__ void particle_pose(const VolumeDesc &V, const FitParams &fp, int i, float R[9], float t[3])
{
    Pose P;
    float d[6];
#pragma unroll
    for (int a = 0; a < 6; ++a)
        d[a] = fp.r[a] * __ldg(&fp.pst[(size_t)a * fp.ld + i]);
    compose_offset(fp.c, d, fp.right_mult != 0, P);
    quat_rot(P.q, R);
    const float s = V.inv_voxel;
#pragma unroll
    for (int a = 0; a < 9; ++a)
        R[a] *= s;
#pragma unroll
    for (int a = 0; a < 3; ++a)
        t[a] = fmaf(P.t[a], s, V.goff[a]);
}

// Points of a unit staged for the pair loop: every coordinate twice, so that one
// 16-byte and one 8-byte broadcast load give the (x, x), (y, y), (z, z) operands.
struct PairPoints {
    ulonglong2 xy[CHUNK_MAX];
    f2_t z[CHUNK_MAX];
};

// Grid-space poses of a lane's two particles, component by component.
struct PairPose {
    f2_t R[9], t[3];
};

// psi of points j .. j + N - 1 for both particles of a lane.  What bounds it on a
// GB300: the FP32 pipe (a .f32x2 instruction holds it two clocks, so pairs save issue
// slots, not arithmetic: 56 instructions a lookup against 80 for the scalar loop of one
// particle per lane, 61 of 124 clocks a scheduler in use) and, for wide swarms, the
// lines a warp's loads touch (one a clock).  All class bytes are loaded, then all
// records, then used.  Three ways through, by warp vote, since a
// wide swarm spends most of its lookups in constant bricks and a converged one
// none: every lookup constant (no record, psi = 1), every lookup mixed (plain
// loads), or both (loads predicated on the class).  321 M lookups of a converged / a
// mixed / a wide swarm (int16, 20,000 particles, sorted) take 0.77 / 0.83 / 0.91 ms
// against 1.08 / 1.19 / 1.18 ms for the scalar loop.  `live` of the points count as
// lookups (the rest repeat the last one).
template <int DT, int N>
__device__ __forceinline__ void pair_lookups(const CellView &V, const PairPoints &sp, int j, int last, int live,
                                             const PairPose &P, f2_t psi[N], int &nva, int &nvb)
{
    const f2_t MAGIC = f2_pack(FLOOR_MAGIC, FLOOR_MAGIC);
    f2_t FX[N], FY[N], FZ[N];
    unsigned ra[N], rb[N];
    int ca[N], cb[N], any = 0, all = -1;
#pragma unroll
    for (int u = 0; u < N; ++u) {
        const int q = min(j + u, last);
        const ulonglong2 xy = sp.xy[q];
        const f2_t X = xy.x, Y = xy.y, Z = sp.z[q];
        const f2_t GX = f2_fma(P.R[0], X, f2_fma(P.R[1], Y, f2_fma(P.R[2], Z, P.t[0])));
        const f2_t GY = f2_fma(P.R[3], X, f2_fma(P.R[4], Y, f2_fma(P.R[5], Z, P.t[1])));
        const f2_t GZ = f2_fma(P.R[6], X, f2_fma(P.R[7], Y, f2_fma(P.R[8], Z, P.t[2])));
        const f2_t TX = f2_add_rd(GX, MAGIC), TY = f2_add_rd(GY, MAGIC), TZ = f2_add_rd(GZ, MAGIC);
        FX[u] = f2_sub(GX, f2_sub(TX, MAGIC));
        FY[u] = f2_sub(GY, f2_sub(TY, MAGIC));
        FZ[u] = f2_sub(GZ, f2_sub(TZ, MAGIC));
        float xa, xb, ya, yb, za, zb;
        f2_unpack(TX, xa, xb);
        f2_unpack(TY, ya, yb);
        f2_unpack(TZ, za, zb);
        ra[u] = cell_record(V, xa, ya, za);
        rb[u] = cell_record(V, xb, yb, zb);
        ca[u] = __ldg(V.cls + (ra[u] >> 9));
        cb[u] = __ldg(V.cls + (rb[u] >> 9));
    }
#pragma unroll
    for (int u = 0; u < N; ++u) {
        any |= ca[u] | cb[u];
        all &= ca[u] & cb[u];
    }
    if (__any_sync(0xffffffffu, any < 0)) {
        CellData<DT> da[N], db[N];
        if (__all_sync(0xffffffffu, all < 0)) {
#pragma unroll
            for (int u = 0; u < N; ++u) {
                cell_fetch<DT, false>(V, ra[u], 0, da[u]);
                cell_fetch<DT, false>(V, rb[u], 0, db[u]);
            }
        } else {
#pragma unroll
            for (int u = 0; u < N; ++u) {
                cell_fetch<DT, true>(V, ra[u], ca[u], da[u]);
                cell_fetch<DT, true>(V, rb[u], cb[u], db[u]);
                nva += u < live ? max(ca[u], 0) : 0;  // free space is valid
                nvb += u < live ? max(cb[u], 0) : 0;
            }
        }
#pragma unroll
        for (int u = 0; u < N; ++u) {
            bool oka, okb;
            psi[u] = cell_eval<DT>(FX[u], FY[u], FZ[u], da[u], db[u], oka, okb);
            nva += (oka && u < live) ? 1 : 0;
            nvb += (okb && u < live) ? 1 : 0;
        }
    } else {
#pragma unroll
        for (int u = 0; u < N; ++u) {
            psi[u] = 0x3F8000003F800000ull;
            nva += u < live ? ca[u] : 0;
            nvb += u < live ? cb[u] : 0;
        }
    }
}

// One lane scores particles ia and ib over the staged points [0, cnt):
// S = sum psi^2 (|psi| with L1), psi = 1 for invalid samples.  Both particles go
// through the same operations side by side, so a particle's sum does not depend
// on its partner.  G terms are added plainly (a partial of <= G terms in [0, 1]),
// then joined to the total with compensation.
template <int DT, int MODE, int G, bool L1>
__device__ __forceinline__ void fitness_pair(const VolumeDesc &Vd, const PairPoints &sp, int cnt, const FitParams &fp,
                                             int ia, int ib, double S_out[2], int n_out[2])
{
    // points in flight at once (a float record takes 8 registers: 3 in flight spill,
    // 454 against 398 us for 9973 particles x 8.4 k points)
    constexpr int N = DT == RF_F32 ? 2 : G / 2;
    static_assert(G % N == 0, "whole batches per group");
    PairPose P;
    {
        float R[2][9], t[2][3];
#pragma unroll
        for (int h = 0; h < 2; ++h)
            particle_pose(Vd, fp, h ? ib : ia, R[h], t[h]);
#pragma unroll
        for (int a = 0; a < 9; ++a)
            P.R[a] = f2_pack(R[0][a], R[1][a]);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            P.t[a] = f2_pack(t[0][a], t[1][a]);
    }
    const CellView V(Vd);
    float sum[2] = {0.f, 0.f}, comp[2] = {0.f, 0.f};
    int nv[2] = {0, 0};
    auto add = [&](float a, float b) {
        if (Mode<MODE>::plain) {
            sum[0] += a;
            sum[1] += b;
        } else {
            neumaier_add(sum[0], comp[0], a);
            neumaier_add(sum[1], comp[1], b);
        }
    };
    int j = 0;
    for (; j + G <= cnt; j += G) {
        f2_t grp = 0ull;
#pragma unroll
        for (int h = 0; h < G; h += N) {
            f2_t psi[N];
            pair_lookups<DT, N>(V, sp, j + h, cnt - 1, N, P, psi, nv[0], nv[1]);
#pragma unroll
            for (int u = 0; u < N; ++u)
                grp = L1 ? f2_add(grp, psi[u] & 0x7FFFFFFF7FFFFFFFull) : f2_fma(psi[u], psi[u], grp);
        }
        float a, b;
        f2_unpack(grp, a, b);
        add(a, b);
    }
    for (; j < cnt; j += N) {  // the tail: term by term
        f2_t psi[N];
        pair_lookups<DT, N>(V, sp, j, cnt - 1, cnt - j, P, psi, nv[0], nv[1]);
#pragma unroll
        for (int u = 0; u < N; ++u)
            if (j + u < cnt) {
                float a, b;
                f2_unpack(L1 ? psi[u] & 0x7FFFFFFF7FFFFFFFull : f2_mul(psi[u], psi[u]), a, b);
                add(a, b);
            }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        S_out[h] = (double)sum[h] + (double)comp[h];
        n_out[h] = nv[h];
    }
}

// Nearest-voxel lookups of one particle over the staged points.
template <int DT, int MODE>
__device__ __forceinline__ void fitness_nearest(const VolumeDesc &Vd, const PairPoints &sp, int cnt, const FitParams &fp,
                                                int i, double &S_out, int &n_out)
{
    float R[9], t[3];
    particle_pose(Vd, fp, i, R, t);
    const CellView V(Vd);
    float sum = 0.f, comp = 0.f;
    int nv = 0;
    for (int j = 0; j < cnt; ++j) {
        const ulonglong2 xy = sp.xy[j];
        const float x = __uint_as_float((unsigned)xy.x), y = __uint_as_float((unsigned)xy.y),
                    z = __uint_as_float((unsigned)sp.z[j]);
        float psi;
        const bool ok = sample_nearest_g<DT>(V, fmaf(R[0], x, fmaf(R[1], y, fmaf(R[2], z, t[0]))),
                                             fmaf(R[3], x, fmaf(R[4], y, fmaf(R[5], z, t[1]))),
                                             fmaf(R[6], x, fmaf(R[7], y, fmaf(R[8], z, t[2]))), psi);
        nv += ok ? 1 : 0;
        psi = ok ? psi : 1.f;
        const float term = fp.l1 ? fabsf(psi) : psi * psi;
        if (Mode<MODE>::plain)
            sum += term;
        else
            neumaier_add(sum, comp, term);
    }
    S_out = (double)sum + (double)comp;
    n_out = nv;
}

// Point j of a unit, staged.
__device__ __forceinline__ void stage_point(PairPoints &sp, int j, const float4 &p)
{
    sp.xy[j] = make_ulonglong2(f2_pack(p.x, p.x), f2_pack(p.y, p.y));
    sp.z[j] = f2_pack(p.z, p.z);
}

// A warp's share of a work unit: 64 particles (two per lane) over the staged points.  Particles beyond the swarm repeat the first one.
template <int DT, int MODE, int G = GROUP>
__device__ __forceinline__ void fitness_unit(const VolumeDesc &V, const PairPoints &sp, int cnt, const FitParams &fp,
                                             const int i[2], double S[2], int nv[2])
{
    const int ia = i[0] < fp.n ? i[0] : 0, ib = i[1] < fp.n ? i[1] : 0;
    if constexpr (Mode<MODE>::nearest) {
        fitness_nearest<DT, MODE>(V, sp, cnt, fp, ia, S[0], nv[0]);
        fitness_nearest<DT, MODE>(V, sp, cnt, fp, ib, S[1], nv[1]);
    } else if (fp.l1) {
        fitness_pair<DT, MODE, G, true>(V, sp, cnt, fp, ia, ib, S, nv);
    } else {
        fitness_pair<DT, MODE, G, false>(V, sp, cnt, fp, ia, ib, S, nv);
    }
}

// Work decomposition shared by the standalone and the persistent kernels: (point
// chunk, group of GROUP_PARTICLES particles, two per lane of a warp).  Consecutive
// groups share a point chunk, so that neighbouring warps read the same part of the
// volume.
struct Split {
    int groups, n_chunks, chunk;
};

__host__ __device__ inline Split make_split(int n, int m, int total_warps, int max_chunks)
{
    Split s;
    s.groups = (n + GROUP_PARTICLES - 1) / GROUP_PARTICLES;
    const int g32 = (n + 31) / 32;  // the chunk length is chosen for groups of 32 particles
    int want = (UNITS_PER_WARP * total_warps + g32 - 1) / g32;
    int lo = (m + CHUNK_MAX - 1) / CHUNK_MAX;   // staging capacity
    int hi = (m + MIN_CHUNK - 1) / MIN_CHUNK;   // at least MIN_CHUNK points per unit
    if (s.groups * hi < total_warps)  // (1024 particles x 4800 points: 555 -> 521 us a frame)
        hi = (m + SMALL_CHUNK - 1) / SMALL_CHUNK;
    want = want < lo ? lo : want;
    want = want > hi ? hi : want;
    want = want > max_chunks ? max_chunks : want;
    want = want < 1 ? 1 : want;
    s.chunk = (m + want - 1) / want;
    if (s.chunk > CHUNK_MAX)  // only when max_chunks binds
        s.chunk = CHUNK_MAX;
    s.n_chunks = (m + s.chunk - 1) / s.chunk;  // every chunk holds a point
    return s;
}

__host__ inline int max_chunks_for(int n, int m_max, int total_warps)
{
    const int groups = (n + 31) / 32;
    const int a = (UNITS_PER_WARP * total_warps + groups - 1) / groups;
    const int b = (m_max + CHUNK_MAX - 1) / CHUNK_MAX;
    return std::max(1, std::max(std::min(a, (m_max + SMALL_CHUNK - 1) / SMALL_CHUNK), b));
}

// rho of a particle's total (Eq. normallh, or Eq. ourlh without NORMALIZE).
__device__ __forceinline__ float fitness_rho(double S, int nO, float tau, bool normalize)
{
    if (nO <= 0)
        return 0.f;
    const double x = normalize ? S / ((double)tau * (double)nO) : S / (double)tau;
    return expf(-(float)x);
}


inline int sm_count()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}

}  // namespace rf
