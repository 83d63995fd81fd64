// Short-range particle-particle part of the P3M force (the guide's P3M kick algorithm with
// split scale PM_scale and cutoff P3M_cutoff, Ch. Parameters):
//
//   a_SR,i = G m * sum_{j: 0 < r_ij < r_c} g(r_ij / r_s) d_ij / (r_ij^2 + eps^2)^(3/2),
//   g(x) = erfc(x/2) + x/sqrt(pi) exp(-x^2/4),
//
// over the particles of the 27 chaining cells around particle i's cell (n_c >= 3 cells of
// side >= r_c, so each neighbour cell appears once and with the minimum image).
//
// CTAs are one warp each (warps never wait for each other), persistent, and take work items (up to
// 32 particles of one cell, most expensive first) from an atomic cursor.  k_pairs_list is the FP32
// kernel, k_pairs64 the FP64 one; their layouts are described below.
#include <cuda_runtime.h>

#include <cstring>
#include <type_traits>

#include "p3m_device.cuh"
#include "p3m_internal.cuh"

namespace {

constexpr int kTJ = P3M_PAIR_TJ;  // 128
constexpr int kBlocksPerTile = kTJ / 32;
constexpr int kLongChunk = 5;   // FP32 kernel: the list is evaluated every 160 entries
constexpr int kShortChunk = 3;  // the autotuner's other choice
constexpr int kGroup = P3M_PAIR_GROUP;

// Coefficients of the FP64 split factor (the context's gpoly64): g = 1 + r^3 sum_k c[k] tau^k
// (k <= P3M_SPLIT_DEG64), tau = r^2 c[P3M_SPLIT_DEG64 + 1] - 1.
struct GPoly64 {
    double c[P3M_SPLIT_DEG64 + 2];
};

// g(r/r_s) (r^2 + eps^2)^-3/2 for one pair in FP64, g from the FP64 fit (largest error about
// 4e-14 relative): rsqrt and a Horner chain instead of sqrt, a division, erfc and exp, which
// all run on GB300's narrow FP64 pipe.  For r2 = 0 the result is not finite; callers select
// such pairs out.
__device__ __forceinline__ double pair_factor64(double r2, double eps2, const GPoly64 &gp)
{
    const double s = rsqrt(r2 + eps2);
    const double r3 = r2 * (r2 * rsqrt(r2));
    const double tau = fma(r2, gp.c[P3M_SPLIT_DEG64 + 1], -1.0);
    double p = gp.c[P3M_SPLIT_DEG64];
#pragma unroll
    for (int k = P3M_SPLIT_DEG64 - 1; k >= 0; --k) p = fma(p, tau, gp.c[k]);
    const double gval = fma(r3, p, 1.0);
    return gval * (s * s * s);
}

// The FP64 kernel.  A lane holds one particle of the work item; the warp streams the j particles of
// the 27 neighbour cells through shared memory in tiles of up to four 32-slot blocks of the sorted
// order, copied by the bulk-copy (TMA) engine into two alternating buffers (the next tile in
// flight while the current one is used; one mbarrier per buffer; every wait bounded).  It skips a
// block when no lane's particle is within r_c of the block's bounding box, evaluates it without
// per-pair tests when the box lies within r_c of every lane's particle, and otherwise tests each
// pair, skipping j's that no lane accepts.  Absolute coordinates: d = (x_j - x_i) + image, like a
// plain minimum-image difference.
struct Neighbour {
    uint32_t start, end;
    double imx, imy, imz;  // periodic image of the neighbour cell
};

__global__ void __launch_bounds__(32)
    k_pairs64(const double4_16a *__restrict__ rel, const double *__restrict__ pos,
            const float4 *__restrict__ block_box, const uint32_t *__restrict__ cell_start,
            const uint32_t *__restrict__ work, const uint32_t *__restrict__ order,
            const uint32_t *__restrict__ n_work_ptr, P3MGeom g, GPoly64 gp, float rcull2, float rin2,
            const double *__restrict__ acc_in, double *__restrict__ acc_out,
            double *__restrict__ mom, double kfac, const double *__restrict__ kfac_dev,
            uint32_t *__restrict__ counters, unsigned long long *__restrict__ pair_count)
{
    if (kfac_dev) kfac = *kfac_dev;  // graph-replayed steps read the factor from the device
    __shared__ __align__(128) double4_16a sj[2][kTJ];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ Neighbour nbr[27];

    const int lane = threadIdx.x;
    const int64_t n = g.n;
    const uint32_t n_work = *n_work_ptr;
    const double rc2 = g.r_c * g.r_c;
    const double eps2 = g.eps * g.eps;
    const int nc = g.n_c;

    if (lane == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncwarp();
    uint32_t parity = 0u;  // bit b: parity of the next phase of bar[b]
    unsigned long long my_pairs = 0, st_fast = 0, st_tested = 0, st_eval = 0, st_culled = 0,
                       st_tiles = 0, st_empty_tiles = 0;
    bool timed_out = false;

    for (;;) {
        uint32_t slot = 0;
        if (lane == 0) slot = atomicAdd(&counters[0], 1u);
        slot = __shfl_sync(0xffffffffu, slot, 0);
        if (slot >= n_work) break;
        const uint32_t item = order[slot];
        const uint32_t cell = work[2 * (size_t)item];
        const uint32_t first = work[2 * (size_t)item + 1];
        const uint32_t cend = cell_start[cell + 1];
        const int cx = (int)(cell % nc), cy = (int)((cell / nc) % nc), cz = (int)(cell / (nc * nc));
        if (lane < 27) {
            const int ox = lane % 3 - 1, oy = (lane / 3) % 3 - 1, oz = lane / 9 - 1;
            const int ux = cx + ox, uy = cy + oy, uz = cz + oz;  // unwrapped neighbour index
            const int wx = (ux + nc) % nc, wy = (uy + nc) % nc, wz = (uz + nc) % nc;
            const uint32_t nb = ((uint32_t)wz * nc + wy) * nc + wx;
            Neighbour q;
            q.start = cell_start[nb];
            q.end = cell_start[nb + 1];
            if (q.start == q.end) q.start = q.end = 0;  // empty: the tile walk skips it
            const double L = g.box;
            q.imx = ux < 0 ? -L : (ux >= nc ? L : 0.0);
            q.imy = uy < 0 ? -L : (uy >= nc ? L : 0.0);
            q.imz = uz < 0 ? -L : (uz >= nc ? L : 0.0);
            nbr[lane] = q;
        }
        __syncwarp();

        const uint32_t i = first + lane;
        const bool valid = i < cend;
        const uint32_t ii = valid ? i : first;
        const double4_16a xi = rel[ii];
        const double xa = pos[ii], ya = pos[n + ii], za = pos[2 * n + ii];  // absolute, FP64
        double ax = 0.0, ay = 0.0, az = 0.0;

        // Tile sequence over (neighbour nb, first block b); a tile is the blocks [b, b + 4)
        // clipped to the neighbour's range of slots; nb == 27 ends the sequence.
        auto next_tile = [&](int &nb, uint32_t &b) {
            while (nb < 27 && b * 32u >= nbr[nb].end) {
                ++nb;
                if (nb < 27) b = nbr[nb].start >> 5;
            }
        };
        auto issue = [&](int nb, uint32_t b, int to) {
            const uint32_t bend = min(b + kBlocksPerTile, (nbr[nb].end + 31) >> 5);
            const uint32_t j0 = b * 32;
            const uint32_t j1 = min((uint32_t)n, bend * 32);
            const uint32_t bytes = (j1 - j0) * (uint32_t)sizeof(double4_16a);
            mbar_expect_tx(&bar[to], bytes);
            bulk_load(&sj[to][0], rel + j0, bytes, &bar[to]);
        };

        int nb_c = 0;
        uint32_t b_c = nbr[0].start >> 5;
        next_tile(nb_c, b_c);
        int buf = 0;
        if (nb_c < 27 && lane == 0) issue(nb_c, b_c, 0);
        while (nb_c < 27) {
            const uint32_t nstart = nbr[nb_c].start, nend = nbr[nb_c].end;
            const uint32_t bend = min(b_c + kBlocksPerTile, (nend + 31) >> 5);
            int nb_n = nb_c;
            uint32_t b_n = bend;
            next_tile(nb_n, b_n);
            __syncwarp();  // every lane is done with sj[buf ^ 1] before it is refilled
            if (nb_n < 27 && lane == 0) issue(nb_n, b_n, buf ^ 1);
            const bool ok = mbar_wait_bounded(&bar[buf], (parity >> buf) & 1u);
            parity ^= 1u << buf;
            if (__any_sync(0xffffffffu, !ok)) {
                timed_out = true;
                if (nb_n < 27) mbar_wait_bounded(&bar[buf ^ 1], (parity >> (buf ^ 1)) & 1u);
                break;
            }
            const Neighbour &q = nbr[nb_c];
            // d = (x_j - x_i) + image, like a plain minimum-image difference
            const double xs = xi.x, ys = xi.y, zs = xi.z;
            const double ix = q.imx, iy = q.imy, iz = q.imz;
            // particle i in the frame of the block boxes (absolute, image removed)
            const float cxs = (float)(xa - q.imx), cys = (float)(ya - q.imy), czs = (float)(za - q.imz);
            const double4_16a *tile = sj[buf];
            double px = 0, py = 0, pz = 0;
            uint32_t cnt = 0, n_fast = 0, n_tested = 0, n_eval = 0, n_culled = 0;
            for (uint32_t b = b_c; b < bend; ++b) {
                const float4 lo = __ldg(block_box + 2 * b), hi = __ldg(block_box + 2 * b + 1);
                const float ex = fmaxf(fmaxf(lo.x - cxs, cxs - hi.x), 0.0f);
                const float ey = fmaxf(fmaxf(lo.y - cys, cys - hi.y), 0.0f);
                const float ez = fmaxf(fmaxf(lo.z - czs, czs - hi.z), 0.0f);
                const bool near = valid && ex * ex + ey * ey + ez * ez < rcull2;
                if (!__any_sync(0xffffffffu, near)) {
                    ++n_culled;
                    continue;
                }
                // the block's slots that belong to the neighbour cell, as tile offsets
                const uint32_t j0 = max(b * 32, nstart) - b_c * 32;
                const uint32_t j1 = min(b * 32 + 32, nend) - b_c * 32;
                const float fx = fmaxf(cxs - lo.x, hi.x - cxs);
                const float fy = fmaxf(cys - lo.y, hi.y - cys);
                const float fz = fmaxf(czs - lo.z, hi.z - czs);
                if (__all_sync(0xffffffffu, !valid || fx * fx + fy * fy + fz * fz < rin2)) {
                    // the block lies within r_c of every particle of the warp
                    n_fast += j1 - j0;
#pragma unroll 2
                    for (uint32_t j = j0; j < j1; ++j) {
                        const double4_16a qj = tile[j];
                        const double dx = (qj.x - xs) + ix, dy = (qj.y - ys) + iy, dz = (qj.z - zs) + iz;
                        const double r2 = dx * dx + dy * dy + dz * dz;
                        const bool in = valid && r2 > 0.0;
                        double f = pair_factor64(r2, eps2, gp);
                        f = in ? f : 0.0;
                        px += f * dx;
                        py += f * dy;
                        pz += f * dz;
                        cnt += in ? 1u : 0u;
                    }
                    continue;
                }
                n_tested += j1 - j0;
                for (uint32_t j = j0; j < j1; ++j) {
                    const double4_16a qj = tile[j];
                    const double dx = (qj.x - xs) + ix, dy = (qj.y - ys) + iy, dz = (qj.z - zs) + iz;
                    const double r2 = dx * dx + dy * dy + dz * dz;
                    const bool in = valid && r2 < rc2 && r2 > 0.0;
                    if (!__any_sync(0xffffffffu, in)) continue;
                    ++n_eval;
                    double f = pair_factor64(r2, eps2, gp);
                    f = in ? f : 0.0;
                    px += f * dx;
                    py += f * dy;
                    pz += f * dz;
                    cnt += in ? 1u : 0u;
                }
            }
            ax += (double)px;
            ay += (double)py;
            az += (double)pz;
            my_pairs += cnt;
            st_fast += n_fast;
            st_tested += n_tested;
            st_eval += n_eval;
            st_culled += n_culled;
            ++st_tiles;
            if (n_culled == bend - b_c) ++st_empty_tiles;
            buf ^= 1;
            nb_c = nb_n;
            b_c = b_n;
        }
        if (timed_out) break;
        if (valid) {
            const double a3[3] = {g.gm * ax, g.gm * ay, g.gm * az};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const double tot = (acc_in ? acc_in[d * n + i] : 0.0) + a3[d];
                acc_out[d * n + i] = tot;
                if (kfac != 0.0) mom[d * n + i] = __dadd_rn(mom[d * n + i], __dmul_rn(kfac, tot));
            }
        }
        __syncwarp();  // nbr is rewritten by the next item
    }
    if (timed_out && lane == 0) atomicOr(&counters[1], P3M_FLAG_TIMEOUT);
    // pair count: warp sum, one atomic per warp
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) my_pairs += __shfl_down_sync(0xffffffffu, my_pairs, o);
    if (lane == 0) {
        if (my_pairs) {
            atomicAdd(pair_count, my_pairs);
            atomicAdd(pair_count + 1, my_pairs);
        }
        if (st_fast) atomicAdd(pair_count + 2, st_fast);
        if (st_tested) atomicAdd(pair_count + 3, st_tested);
        if (st_eval) atomicAdd(pair_count + 4, st_eval);
        if (st_culled) atomicAdd(pair_count + 5, st_culled);
        if (st_tiles) atomicAdd(pair_count + 6, st_tiles);
        if (st_empty_tiles) atomicAdd(pair_count + 7, st_empty_tiles);
    }
}

// ------------------------------------------------------------------ FP32 mode, compacted j lists
// The FP32 kernel.  A work item's up to 32 particles are taken in groups of kG (consecutive along
// the Hilbert order inside the cell, so compact), one group at a time per one-warp CTA:
//   1. The neighbour cells form 9 rows of 3 along x, each a contiguous range of sorted slots (two
//      ranges where a row wraps).  The rows' 32-slot blocks are tested 32 at a time, one per lane,
//      against the group's bounding box (block_box, padded by more than its FP32 rounding).
//   2. Lane l of the warp holds slot l of a surviving block and tests that one particle against
//      the group's box; the accepted ones are appended to a list in shared memory (ballot and
//      prefix count), as coordinates relative to the group's centre.
//   3. Every 32 kChunkBlocks entries the list is evaluated: a lane owns two particles i and takes
//      every (64/kG)-th pair of consecutive entries, two entries at once in packed f32x2
//      arithmetic, so that one 8-byte load per coordinate serves four pair slots.
// Before, 32 particles met every j of the tested blocks, one particle per lane: 37 % of the
// evaluated lane slots held an accepted pair at 200 particles per cell, and half of the
// instructions were tests and votes.  The list holds 47 % accepted slots at kG = 16 (58 % at 8,
// 39 % at 32: the union of the cutoff spheres grows with the group), there are no votes between
// pairs, and a test sequence serves 32 candidates of the whole group.  Measured at 128^3 (one
// evaluation, before / after): near-uniform 5.23 / 3.12 ms, clustered 12.3 / 9.6 ms.
// What bounds it now: of 81 cycles per 32 accepted pairs and scheduler, 55 are the evaluation
// (26 per 32 slots; two FP32 operations with three distinct registers already take three cycles
// of register bandwidth, and the same mix of 16 packed operations, 2 rsqrt and 2 ex2 alone runs
// at 20.5), 20 the candidate tests and 6 the set-up of groups.  16 particles per group
// and 18 CTAs per SM: 8, 32 and 16, 20, 24 are within 3 % or slower on both sets.
//
// Coordinates are 32-bit fixed point, 2^-29 of a chaining cell, modulo 8 cells (relq): differences
// of particles in neighbouring cells, periodic images included, are exact integers, and only the
// difference from the group's centre is rounded to FP32 and scaled (PairFactor).
//
// A pair at r = 0 (the particle itself, or a coincident one) gets a finite factor (r^2 starts at
// kTinyQ when there is no softening) and contributes exactly f * 0.  Only the row of the own cell
// can hold such pairs; there (kOwn) a pair counts only if one of its differences is non-zero.

constexpr int kPairSegs = 18;           // 9 rows of neighbour cells, each at most two ranges
constexpr int kFlushTerms = 80;         // FP32 terms per partial sum before it joins the FP64 sum
constexpr float kTinyQ = 1e-24f;        // far below the smallest non-zero scaled r^2
constexpr float kFarQ = 1e6f;           // scaled coordinate of a padding entry: outside every cutoff

// One range of neighbour slots of a group: its slots, the group's centre in the range's periodic
// image (fixed point, and absolute FP32 for the block boxes), and the number of blocks before it.
struct __align__(16) PairSeg {
    uint32_t start, end, cx, cy;
    uint32_t cz, first_block;
    float ax, ay;
    float az, pad[3];
};

struct PairConstQ {
    f2 c[5];
    f2 na, ab, e2, tiny;
};

// The factor g(r/r_s) (r^2 + eps^2)^-3/2 of both halves of w (see PairFactor and fit_pair_factor).
// The MUFU pipe takes 8 cycles per warp for a reciprocal or a square root, so that the former
// rsqrt, rcp and sqrt per pair cost as much as 24 FP32 operations; here it is one rsqrt and one
// ex2.  kAdditive (softening small against r_s): 16 FP32 operations per pair with the distance
// and the accumulation; otherwise 21 and one more rsqrt.
template <bool kAdditive>
__device__ __forceinline__ f2 pair_factor_q(f2 w, const PairConstQ &k)
{
    float wl, wh;
    f2_unpack(w, wl, wh);
    const f2 t = f2_pack(ex2_approx(-wl), ex2_approx(-wh));
    const f2 rw = f2_pack(rsqrt_approx(wl), rsqrt_approx(wh));
    f2 p = kAdditive ? k.c[3] : f2_fma(k.c[4], t, k.c[3]);
    p = f2_fma(p, t, k.c[2]);
    p = f2_fma(p, t, k.c[1]);
    if (kAdditive) {
        const f2 q = f2_fma(k.na, t, f2_add(rw, k.ab));
        return f2_fma(p, t, f2_fma(q, f2_mul(rw, rw), k.c[0]));
    }
    p = f2_fma(p, t, k.c[0]);
    float sl, sh;
    f2_unpack(f2_add(w, k.e2), sl, sh);
    const f2 s = f2_pack(rsqrt_approx(sl), rsqrt_approx(sh));
    const f2 m = f2_fma(w, p, f2_fma(k.na, t, k.ab));
    const f2 gv = f2_fma(f2_mul(w, rw), m, f2_pack(1.0f, 1.0f));
    return f2_mul(f2_mul(gv, s), f2_mul(s, s));
}

// kForm: 1 the additive factor, 0 the general one, 2 each context's own (batched launches)
template <bool kBatched, int kForm, int kChunkBlocks, int kG>
__global__ void __launch_bounds__(32, P3M_PAIR_CTAS)
    k_pairs_list(PairArgs a0, const PairArgs *__restrict__ descs, const uint32_t *__restrict__ order,
                 const uint32_t *__restrict__ n_work_ptr, uint32_t *__restrict__ cursor)
{
    constexpr int kArgWords = sizeof(PairArgs) / 8;
    static_assert(sizeof(PairArgs) % 8 == 0, "PairArgs is copied in 8-byte words");
    constexpr int kChunk = 32 * kChunkBlocks, kCap = kChunk + 32;
    constexpr int kPairsI = kG / 2;        // lanes that share one list entry
    constexpr int kStride = 2 * (32 / kPairsI);  // list entries per warp step
    constexpr int kSub = P3M_PAIR_TI / kG;
    constexpr int kFlushChunks = kFlushTerms * kStride / kChunk < 1 ? 1 : kFlushTerms * kStride / kChunk;
    static_assert(kChunk % kStride == 0, "whole steps per chunk");
    __shared__ __align__(16) float list[3][kCap];
    __shared__ double sum[6][32];  // per lane: x, y, z of its first particle, then of its second
    __shared__ PairSeg seg[kPairSegs];
    __shared__ uint32_t live[32];
    __shared__ unsigned long long stat[6];
    __shared__ __align__(16) PairArgs sA;  // the current work item's context
    const PairArgs &A = sA;

    const int lane = threadIdx.x;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t n_units = *n_work_ptr * kSub;
    const int ip = lane % kPairsI, js = lane / kPairsI;
    int cur_sim = -1;
    double kfac = 0.0;
    PairConstQ kc;
    // (re)load the context's arguments into shared memory and the per-lane constants
    auto load_args = [&](const PairArgs *src) {
        __syncwarp();  // every lane is done with the previous arguments
        const uint64_t *from = (const uint64_t *)src;
        uint64_t *to = (uint64_t *)&sA;
        for (int w = lane; w < kArgWords; w += 32) to[w] = from[w];
        if (lane < 6) stat[lane] = 0ull;
        __syncwarp();
        kfac = A.kfac_dev ? *A.kfac_dev : A.kfac;
#pragma unroll
        for (int q = 0; q < 5; ++q) kc.c[q] = f2_pack(A.fac.c[q], A.fac.c[q]);
        kc.na = f2_pack(A.fac.na, A.fac.na);
        kc.ab = f2_pack(A.fac.ab, A.fac.ab);
        kc.e2 = f2_pack(A.fac.e2, A.fac.e2);
        kc.tiny = f2_pack(kTinyQ, kTinyQ);
    };
    // the counters gathered so far, into their context
    auto store_stat = [&]() {
        __syncwarp();
        if (lane < 6 && stat[lane]) {
            atomicAdd(A.pair_count + lane + (lane ? 2 : 1), stat[lane]);
            if (lane == 0) atomicAdd(A.pair_count, stat[0]);
        }
    };
    if (!kBatched) load_args(&a0);

    for (;;) {
        uint32_t unit = 0;
        if (lane == 0) unit = atomicAdd(cursor, 1u);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= n_units) break;
        uint32_t item = order[unit / kSub];
        if (kBatched) {
            const int sim = (int)(item >> 24);
            item &= 0xFFFFFFu;
            if (sim != cur_sim) {
                if (cur_sim >= 0) store_stat();
                load_args(descs + sim);
                cur_sim = sim;
            }
        }
        const P3MGeom &g = A.g;
        const int64_t n = g.n;
        const int nc = g.n_c;
        const uint32_t cell = A.work[2 * (size_t)item];
        const uint32_t first = A.work[2 * (size_t)item + 1] + (unit % kSub) * kG;
        const uint32_t cend = A.cell_start[cell + 1];
        if (first >= cend) continue;
        const int cx = (int)(cell % nc), cy = (int)((cell / nc) % nc), cz = (int)(cell / (nc * nc));

        // the group's bounding box around an integer centre; lane l < kG holds particle l
        uint32_t ctr[3];
        float half[3], actr[3];
        {
            const uint32_t i = min(first + min(lane, kG - 1), cend - 1);
            const uint32_t *q = A.relq + (size_t)(i >> 5) * 96 + (i & 31);
            const int c3[3] = {cx, cy, cz};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const uint32_t x = __ldg(q + 32 * d), x0 = __shfl_sync(0xffffffffu, x, 0);
                const int lo = __reduce_min_sync(0xffffffffu, (int)(x - x0));
                const int hi = __reduce_max_sync(0xffffffffu, (int)(x - x0));
                const int mid = lo + ((hi - lo) >> 1);
                ctr[d] = x0 + (uint32_t)mid;
                half[d] = (float)(max(hi - mid, mid - lo)) * (1.0f + 0x1p-20f) * A.fac.lambda;
                // absolute FP32 centre: cell index and offset inside the cell, in cell sides
                actr[d] = ((float)c3[d] + (float)(int)(ctr[d] - ((uint32_t)c3[d] << kFixBits)) * kFixUnit) *
                          A.fac.cell;
            }
        }
        __syncwarp();  // the previous group is done with seg
        uint32_t nblk = 0;
        if (lane < kPairSegs) {
            const int row = ((lane >> 1) + 4) % 9;  // the own row (4) comes first
            const int uy = cy + row % 3 - 1, uz = cz + row / 3 - 1;
            const int wy = uy < 0 ? uy + nc : (uy >= nc ? uy - nc : uy);
            const int wz = uz < 0 ? uz + nc : (uz >= nc ? uz - nc : uz);
            const int iy = uy < 0 ? -1 : (uy >= nc ? 1 : 0), iz = uz < 0 ? -1 : (uz >= nc ? 1 : 0);
            int x0 = max(cx - 1, 0), x1 = min(cx + 1, nc - 1), ix = 0;
            if (lane & 1) {  // the wrapped end of the row, if any
                ix = cx == 0 ? -1 : (cx == nc - 1 ? 1 : 0);
                x0 = x1 = cx == 0 ? nc - 1 : 0;
            }
            const uint32_t base = ((uint32_t)wz * nc + wy) * nc;
            uint32_t s = A.cell_start[base + x0], e = A.cell_start[base + x1 + 1];
            if (!p3m_in_bounds(s <= e && e <= (uint32_t)n, g.flags)) e = s;
            if ((lane & 1) && ix == 0) e = s;
            PairSeg q;
            q.start = s;
            q.end = e;
            const uint32_t box = (uint32_t)nc << kFixBits;  // the box side modulo 2^32
            q.cx = ctr[0] - (uint32_t)ix * box;
            q.cy = ctr[1] - (uint32_t)iy * box;
            q.cz = ctr[2] - (uint32_t)iz * box;
            q.ax = actr[0] - (float)(ix * nc) * A.fac.cell;
            q.ay = actr[1] - (float)(iy * nc) * A.fac.cell;
            q.az = actr[2] - (float)(iz * nc) * A.fac.cell;
            nblk = e > s ? ((e - 1) >> 5) - (s >> 5) + 1 : 0;
            uint32_t incl = nblk;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync((1u << kPairSegs) - 1u, incl, o);
                if (lane >= o) incl += y;
            }
            q.first_block = incl - nblk;
            seg[lane] = q;
            nblk = incl;
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) sum[q][lane] = 0.0;
        __syncwarp();
        const uint32_t own_blocks = __shfl_sync(0xffffffffu, nblk, 1);
        const uint32_t all_blocks = __shfl_sync(0xffffffffu, nblk, kPairSegs - 1);

        // the lane's two particles, relative to the centre and negated
        const float lambda = A.fac.lambda;
        f2 nx[2], ny[2], nz[2], px[2], py[2], pz[2];
        uint32_t cnt[2] = {0u, 0u};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint32_t i = min(first + ip + u * kPairsI, cend - 1);
            const uint32_t *q = A.relq + (size_t)(i >> 5) * 96 + (i & 31);
            const float x = (float)(int)(__ldg(q) - ctr[0]) * -lambda,
                        y = (float)(int)(__ldg(q + 32) - ctr[1]) * -lambda,
                        z = (float)(int)(__ldg(q + 64) - ctr[2]) * -lambda;
            nx[u] = f2_pack(x, x);
            ny[u] = f2_pack(y, y);
            nz[u] = f2_pack(z, z);
            px[u] = py[u] = pz[u] = f2_pack(0.0f, 0.0f);
        }
        const float rc2 = A.fac.rc2, rlist2 = A.fac.rlist2;
        const uint32_t *__restrict__ relq = A.relq + lane;

        auto flush = [&]() {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                sum[3 * u][lane] += (double)(px[u].x + px[u].y);
                sum[3 * u + 1][lane] += (double)(py[u].x + py[u].y);
                sum[3 * u + 2][lane] += (double)(pz[u].x + pz[u].y);
                px[u] = py[u] = pz[u] = f2_pack(0.0f, 0.0f);
            }
        };
        // list entries [0, count), count a multiple of kStride
        auto eval_form = [&](auto additive, auto own, int count) {
            constexpr bool kAdd = decltype(additive)::value;
            const f2 w0 = kAdd ? kc.e2 : kc.tiny;
            const float *lx = &list[0][2 * js], *ly = &list[1][2 * js], *lz = &list[2][2 * js];
            f2 Xn = *(const f2 *)lx, Yn = *(const f2 *)ly, Zn = *(const f2 *)lz;
#pragma unroll 1
            for (int k = 0; k < count; k += kStride) {
                const f2 X = Xn, Y = Yn, Z = Zn;
                const int kn = k + kStride < count ? k + kStride : 0;
                Xn = *(const f2 *)(lx + kn), Yn = *(const f2 *)(ly + kn), Zn = *(const f2 *)(lz + kn);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const f2 dx = f2_add(X, nx[u]), dy = f2_add(Y, ny[u]), dz = f2_add(Z, nz[u]);
                    const f2 w = f2_fma(dz, dz, f2_fma(dy, dy, f2_fma(dx, dx, w0)));
                    f2 f = pair_factor_q<kAdd>(w, kc);
                    const bool lo = w.x < rc2, hi = w.y < rc2;
                    f.x = lo ? f.x : 0.0f;
                    f.y = hi ? f.y : 0.0f;
                    px[u] = f2_fma(f, dx, px[u]);
                    py[u] = f2_fma(f, dy, py[u]);
                    pz[u] = f2_fma(f, dz, pz[u]);
                    if (decltype(own)::value) {
                        const bool nl = (__float_as_uint(dx.x) | __float_as_uint(dy.x) | __float_as_uint(dz.x)) != 0u;
                        const bool nh = (__float_as_uint(dx.y) | __float_as_uint(dy.y) | __float_as_uint(dz.y)) != 0u;
                        if (lo && nl) ++cnt[u];
                        if (hi && nh) ++cnt[u];
                    } else {
                        if (lo) ++cnt[u];
                        if (hi) ++cnt[u];
                    }
                }
            }
        };
        auto eval = [&](auto own, int count) {
            if (kForm == 1 || (kForm == 2 && A.fac.additive))
                eval_form(std::true_type{}, own, count);
            else
                eval_form(std::false_type{}, own, count);
        };

        uint32_t n_list = 0, n_live = 0, n_chunks = 0;
        int fill = 0;
        // the blocks [t0, t1) of the ranges in sequence
        auto walk = [&](auto own, uint32_t t0, uint32_t t1) {
            for (uint32_t base = t0; base < t1; base += 32) {
                const uint32_t t = base + lane;
                bool keep = false;
                uint32_t word = 0;
                if (t < t1) {
                    int s = 0;  // the last range that starts at or before block t
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
                        if (s + o < kPairSegs && seg[s + o].first_block <= t) s += o;
                    const uint32_t b = (seg[s].start >> 5) + (t - seg[s].first_block);
                    const float4 lo = __ldg(A.block_box + 2 * (size_t)b), hi = __ldg(A.block_box + 2 * (size_t)b + 1);
                    const float hx = half[0] * A.fac.length, hy = half[1] * A.fac.length, hz = half[2] * A.fac.length;
                    const float ex = fmaxf(fmaxf(lo.x - seg[s].ax, seg[s].ax - hi.x) - hx, 0.0f);
                    const float ey = fmaxf(fmaxf(lo.y - seg[s].ay, seg[s].ay - hi.y) - hy, 0.0f);
                    const float ez = fmaxf(fmaxf(lo.z - seg[s].az, seg[s].az - hi.z) - hz, 0.0f);
                    keep = ex * ex + ey * ey + ez * ez < A.rcull2;
                    word = ((uint32_t)s << 26) | b;
                }
                const uint32_t m = __ballot_sync(0xffffffffu, keep);
                if (keep) live[__popc(m & lt)] = word;
                __syncwarp();
                const int nl = __popc(m);
                n_live += nl;
                // the next block's coordinates are loaded while the current one is tested
                uint32_t word_n = 0, xn = 0, yn = 0, zn = 0;
                auto fetch = [&](int k) {
                    word_n = live[k];
                    const uint32_t *q = relq + (size_t)(word_n & 0x3FFFFFFu) * 96;
                    xn = __ldg(q);
                    yn = __ldg(q + 32);
                    zn = __ldg(q + 64);
                };
                if (nl) fetch(0);
#pragma unroll 1
                for (int k = 0; k < nl; ++k) {
                    const PairSeg &S = seg[word_n >> 26];
                    const uint32_t slot = (word_n & 0x3FFFFFFu) * 32 + lane;
                    const float x = (float)(int)(xn - S.cx) * lambda, y = (float)(int)(yn - S.cy) * lambda,
                                z = (float)(int)(zn - S.cz) * lambda;
                    const bool mine = slot - S.start < S.end - S.start;
                    if (k + 1 < nl) fetch(k + 1);
                    const float ex = fmaxf(fabsf(x) - half[0], 0.0f), ey = fmaxf(fabsf(y) - half[1], 0.0f),
                                ez = fmaxf(fabsf(z) - half[2], 0.0f);
                    const bool in = mine && ex * ex + ey * ey + ez * ez < rlist2;
                    const uint32_t mm = __ballot_sync(0xffffffffu, in);
                    if (in) {
                        const int p = fill + __popc(mm & lt);
                        list[0][p] = x;
                        list[1][p] = y;
                        list[2][p] = z;
                    }
                    fill += __popc(mm);
                    if (fill >= kChunk) {
                        __syncwarp();
                        eval(own, kChunk);
                        __syncwarp();
                        fill -= kChunk;
                        if (lane < fill) {  // (reads and writes do not overlap: fill < 32 <= kChunk)
                            list[0][lane] = list[0][kChunk + lane];
                            list[1][lane] = list[1][kChunk + lane];
                            list[2][lane] = list[2][kChunk + lane];
                        }
                        n_list += kChunk;
                        if (++n_chunks % kFlushChunks == 0) flush();
                    }
                }
                __syncwarp();  // live is rewritten by the next 32 blocks
            }
            // the rest of the list, padded to whole steps with far entries
            const int count = (fill + kStride - 1) / kStride * kStride;
            if (lane < count - fill) list[0][fill + lane] = list[1][fill + lane] = list[2][fill + lane] = kFarQ;
            __syncwarp();
            eval(own, count);
            __syncwarp();
            flush();
            n_list += fill;
            fill = 0;
        };
        walk(std::true_type{}, 0u, own_blocks);
        walk(std::false_type{}, own_blocks, all_blocks);
        __syncwarp();

        // particle t of the group: the sums of the 32/kPairsI lanes that shared it, in lane order
        const double *__restrict__ acc_in = A.acc_in;
        double *__restrict__ acc_out = A.acc_out;
        double *__restrict__ mom = A.mom;
        for (int t = lane; t < 3 * kG; t += 32) {
            const int d = t / kG, k = t % kG;
            const uint32_t i = first + k;
            if (i >= cend) continue;
            double s = 0.0;
#pragma unroll
            for (int o = 0; o < 32 / kPairsI; ++o) s += sum[3 * (k / kPairsI) + d][o * kPairsI + k % kPairsI];
            const double tot = (acc_in ? acc_in[d * n + i] : 0.0) + A.fac.scale * s;
            acc_out[d * n + i] = tot;
            if (kfac != 0.0) mom[d * n + i] = __dadd_rn(mom[d * n + i], __dmul_rn(kfac, tot));
        }
        // the group's pair count and work counters
        const uint32_t my = (first + ip < cend ? cnt[0] : 0u) + (first + ip + kPairsI < cend ? cnt[1] : 0u);
        const uint32_t pairs = __reduce_add_sync(0xffffffffu, my);
        if (lane == 0) {
            stat[0] += pairs;
            stat[1] += (n_live * kG);              // j's tested against the group's box, in slots of 32
            stat[2] += (n_list * kG + 16) / 32;    // list entries evaluated, the same
            stat[3] += all_blocks - n_live;
            stat[4] += n_chunks + 2;
        }
        __syncwarp();
    }
    if (!kBatched || cur_sim >= 0) store_stat();
}

cudaError_t pairs64_impl(p3m_ctx *c, const double *acc_in, double *acc_out, double kfac,
                       const double *kfac_dev)
{
    cudaMemsetAsync(c->counters, 0, sizeof(uint32_t), c->stream);
    cudaMemsetAsync(c->pair_count, 0, sizeof(unsigned long long), c->stream);  // last evaluation
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pairs64, 32, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const int grid = c->num_sms * per_sm;
    GPoly64 gp;
    for (int k = 0; k < P3M_SPLIT_DEG64 + 2; ++k) gp.c[k] = c->gpoly64[k];
    // culling radii: r_c widened (narrowed) by more than the FP32 rounding of absolute
    // coordinates up to the box size
    const double rcull = c->g.r_c * (1.0 + 1e-4) + c->g.box * 1e-6;
    const double rin = c->g.r_c * (1.0 - 1e-4) - c->g.box * 1e-6;
    c->launches += 1;
    k_pairs64<<<grid, 32, 0, c->stream>>>(
        (const double4_16a *)c->rel, c->pos, c->block_box, c->cell_start, c->work,
        c->work_order, c->work_off + c->g.n_cells, c->g, gp, (float)(rcull * rcull),
        rin > 0.0 ? (float)(rin * rin) : 0.0f, acc_in, acc_out, c->mom, kfac, kfac_dev,
        c->counters, c->pair_count);
    return cudaGetLastError();
}

// The FP32 kernel for one context or (batched) several.
template <bool kBatched, int kForm, int kChunkBlocks>
cudaError_t launch_list(const PairArgs &a, const PairArgs *descs, const uint32_t *order,
                        const uint32_t *n_work, uint32_t *cursor, int num_sms, cudaStream_t s)
{
    int per_sm = 0;
    auto kern = k_pairs_list<kBatched, kForm, kChunkBlocks, kGroup>;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32, 0);
    if (e != cudaSuccess) return e;
    kern<<<num_sms * (per_sm < 1 ? 1 : per_sm), 32, 0, s>>>(a, descs, order, n_work, cursor);
    return cudaGetLastError();
}

cudaError_t pairs_list_impl(p3m_ctx *c, const double *acc_in, double *acc_out, double kfac,
                            const double *kfac_dev)
{
    cudaMemsetAsync(c->counters, 0, sizeof(uint32_t), c->stream);
    cudaMemsetAsync(c->pair_count, 0, sizeof(unsigned long long), c->stream);  // last evaluation
    c->launches += 1;
    const PairArgs a = pair_args(c, acc_in, acc_out, kfac, kfac_dev);
    const uint32_t *n_work = c->work_off + c->g.n_cells;
    const bool add = c->pair_factor.additive != 0;
    auto launch = c->tile_blocks == kShortChunk ? (add ? launch_list<false, 1, kShortChunk> : launch_list<false, 0, kShortChunk>)
                                                : (add ? launch_list<false, 1, kLongChunk> : launch_list<false, 0, kLongChunk>);
    return launch(a, nullptr, c->work_order, n_work, c->counters, c->num_sms, c->stream);
}

__global__ void k_store_pair_args(PairArgs *dst, PairArgs a) { *dst = a; }

__global__ void k_ens_gather(uint32_t slot, const uint32_t *__restrict__ key,
                             const uint32_t *__restrict__ order, size_t n, uint32_t *__restrict__ gk,
                             uint32_t *__restrict__ gv)
{
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n;
         k += (size_t)gridDim.x * blockDim.x) {
        gk[k] = key[k];
        gv[k] = (slot << 24) | (order[k] & 0xFFFFFFu);
    }
}

__global__ void k_ens_total(const uint32_t *const *nwork, int nb, uint32_t *total)
{
    uint32_t t = 0;
    for (int k = 0; k < nb; ++k) t += *nwork[k];
    *total = t;
}

}  // namespace

PairArgs pair_args(const p3m_ctx *c, const double *acc_in, double *acc_out, double kfac,
                   const double *kfac_dev)
{
    PairArgs a;
    memset(&a, 0, sizeof(a));
    a.relq = c->relq;
    a.block_box = c->block_box;
    a.cell_start = c->cell_start;
    a.work = c->work;
    a.acc_in = acc_in;
    a.acc_out = acc_out;
    a.mom = c->mom;
    a.kfac_dev = kfac_dev;
    a.counters = c->counters;
    a.pair_count = c->pair_count;
    a.kfac = kfac;
    a.g = c->g;
    a.fac = c->pair_factor;
    // culling radius: r_c widened by more than the FP32 rounding of absolute coordinates up to the
    // box size
    const double rcull = c->g.r_c * (1.0 + 1e-4) + c->g.box * 1e-6;
    a.rcull2 = (float)(rcull * rcull);
    return a;
}

cudaError_t launch_pairs_batched(const PairArgs *descs, const uint32_t *order,
                                 const uint32_t *n_total, uint32_t *cursor, int num_sms,
                                 cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(cursor, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    PairArgs unused;
    memset(&unused, 0, sizeof(unused));
    return launch_list<true, 2, kLongChunk>(unused, descs, order, n_total, cursor, num_sms, s);
}

cudaError_t launch_store_pair_args(PairArgs *dst, const PairArgs &a, cudaStream_t s)
{
    k_store_pair_args<<<1, 1, 0, s>>>(dst, a);
    return cudaGetLastError();
}

cudaError_t launch_ens_gather(int slot, const uint32_t *key, const uint32_t *order, size_t n,
                              uint32_t *gkey, uint32_t *gval, cudaStream_t s)
{
    const size_t blocks = (n + 255) / 256;
    k_ens_gather<<<(unsigned)(blocks < 1 ? 1 : (blocks > 1024 ? 1024 : blocks)), 256, 0, s>>>(
        (uint32_t)slot, key, order, n, gkey, gval);
    return cudaGetLastError();
}

cudaError_t launch_ens_total(const uint32_t *const *nwork, int nb, uint32_t *total, cudaStream_t s)
{
    k_ens_total<<<1, 1, 0, s>>>(nwork, nb, total);
    return cudaGetLastError();
}

cudaError_t launch_pairs(p3m_ctx *c, const double *acc_in, double *acc_out, double kfac,
                         const double *kfac_dev)
{
    return c->precision == P3M_PREC_MIXED ? pairs_list_impl(c, acc_in, acc_out, kfac, kfac_dev)
                                          : pairs64_impl(c, acc_in, acc_out, kfac, kfac_dev);
}
