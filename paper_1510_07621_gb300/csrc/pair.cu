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
#include "pair_walk.cuh"

namespace {

constexpr int kLongChunk = 5;   // FP32 kernel: the list is evaluated every 160 entries
constexpr int kShortChunk = 3;  // the autotuner's other choice

// x^-1/2: the hardware's approximation (relative error e0 / 2 below 2^-20) and one step of the
// third-order iteration y (1 + e/2 + 3 e^2/8), e = 1 - x y^2, whose error 5/16 e^3 is below 2^-58.
__device__ __forceinline__ double rsqrt64(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-(x * y), y, 1.0);
    return fma(y * e, fma(e, 0.375, 0.5), y);
}

// g(r/r_s) (r^2 + eps^2)^-3/2 for one pair in FP64.  g comes from the context's table (tab: 64
// intervals of r in [0, r_c], a degree-7 polynomial in t in [-1, 1] each, see fit_split_table): 7
// FP64 operations per pair, where one polynomial over the whole range takes 18 and two to form r^3.
// The interval index needs no FP64 operation: r truncated to FP32 by its bits; at an interval's end it
// may be one off, and t then exceeds 1 by 1e-5.  For r2 = 0 the result is not finite, beyond r_c it is
// extrapolated; callers select such pairs out.
__device__ __forceinline__ double pair_factor64(double r2, double eps2, float scale_f, double scale,
                                                const double *tab)
{
    const double ri = rsqrt64(r2), s = eps2 == 0.0 ? ri : rsqrt64(r2 + eps2);
    const double r = r2 * ri;
    const int hi = __double2hiint(r), e = (hi >> 20 & 0x7FF) - 1023 + 127;
    const float rf = e >= 1 && e <= 254 ? __int_as_float((e << 23) | (hi & 0xFFFFF) << 3) : 0.0f;
    const int k = min((int)(rf * scale_f), kSplitTab64 - 1);
    const double *c = tab + k * kSplitRow64;
    const double t = fma(r, scale, c[8]);  // (c[8] = -(2 k + 1))
    double p = fma(c[7], t, c[6]);
#pragma unroll
    for (int q = 5; q >= 0; --q) p = fma(p, t, c[q]);
    return p * (s * s * s);
}

// The FP64 kernel.  GB300's FP64 pipe issues one warp instruction in 16 cycles per SM, 64 times fewer
// than the FP32 pipes, so that everything but the accepted pairs' arithmetic is kept off it.  A
// one-warp CTA takes 8 particles of a work item at a time, four lanes to a particle:
//   1. For up to kEntries32 surviving 32-slot blocks (pair_walk.cuh) it tests every (particle, slot)
//      in FP32 on the fixed-point coordinates, with a radius padded by more than their rounding, and
//      keeps one 32-bit mask per particle and block in shared memory.
//   2. Lane q of a particle then takes the pairs number q, q + 4, q + 8, ... of its masks: every step
//      evaluates 32 different pairs in FP64 (d = (x_j - x_i) + image, like a plain minimum-image
//      difference, and the exact test 0 < r < r_c), whatever blocks they lie in.
// Before, a lane held one particle and all lanes met the same j, tested in FP64: 0.37 of the
// evaluated and 0.2 of the tested lane slots held an accepted pair, and 32^3 particles gave too few
// warps to hide the FP64 latency.  One step (two evaluations) of 32^3 particles: 38.9 -> 4.6 ms, of
// the clustered 48^3 set 2.9 to 5 times less (more, the more clustered).  What bounds it: the 32 FP64
// operations of a pair (45 before the table of g, 2.0 instead of 2.8 ms per evaluation at 32^3);
// at the measured FP64 rate they take 1.5 ms there.
constexpr int kEntries64 = 96;  // blocks per round (about what a group of 8 has in all at 200 per cell)

__global__ void __launch_bounds__(32)
    k_pairs64(const uint32_t *__restrict__ relq, const double *__restrict__ pos,
              const float4 *__restrict__ block_box, const uint32_t *__restrict__ cell_start,
              const uint32_t *__restrict__ work,
              const uint32_t *__restrict__ n_work_ptr, P3MGeom g, const double *__restrict__ split, float rcull2, float rlist2,
              const double *__restrict__ acc_in, double *__restrict__ acc_out,
              double *__restrict__ mom, double kfac, const double *__restrict__ kfac_dev,
              uint32_t *__restrict__ cursor, unsigned long long *__restrict__ pair_count)
{
    constexpr int kG = 8, kSub = P3M_PAIR_TI / kG;
    if (kfac_dev) kfac = *kfac_dev;  // graph-replayed steps read the factor from the device
    __shared__ uint32_t mask[kEntries64][kG];
    __shared__ uint32_t entry[kEntries64];
    __shared__ __align__(16) float sj[3][32];
    __shared__ PairSeg seg[kPairSegs];
    __shared__ LiveBlocks live;
    __shared__ __align__(16) double tab[kSplitTab64 * kSplitRow64];
    for (int t = threadIdx.x; t < kSplitTab64 * kSplitRow64; t += 32) tab[t] = split[t];
    __syncwarp();

    const int lane = threadIdx.x, pi = lane & 7, q = lane >> 3;  // particle of the group, its lane
    const int64_t n = g.n;
    const uint32_t n_units = *n_work_ptr * kSub;
    const long long rc2 = __double_as_longlong(g.r_c * g.r_c);
    const double eps2 = g.eps * g.eps, tscale = 2.0 * kSplitTab64 / g.r_c;
    const float kscale = (float)(kSplitTab64 / g.r_c);
    const int nc = g.n_c;
    const float cell_f = (float)g.cs;
    unsigned long long st_pairs = 0, st_tested = 0, st_steps = 0, st_culled = 0, st_rounds = 0, st_empty = 0;

    for (;;) {
        uint32_t unit = 0;
        if (lane == 0) unit = atomicAdd(cursor, 1u);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= n_units) break;
        const uint32_t item = unit / kSub;
        const uint32_t cell = work[2 * (size_t)item];
        const uint32_t first = work[2 * (size_t)item + 1] + (unit % kSub) * kG;
        const uint32_t cend = cell_start[cell + 1];
        if (first >= cend) continue;
        const int cx = (int)(cell % nc), cy = (int)((cell / nc) % nc), cz = (int)(cell / (nc * nc));
        // FP32 frame in cell sides
        const GroupFrame fr = group_frame<kG>(relq, first, cend, cx, cy, cz, kFixUnit, cell_f);
        const uint2 blocks = group_ranges(seg, cell_start, g, cx, cy, cz, fr, cell_f);
        const uint32_t i = min(first + pi, cend - 1);
        const bool valid = first + pi < cend;
        const uint32_t *qi = fix_coords(relq, i);
        const float fx = (float)(int)(__ldg(qi) - fr.ctr[0]) * kFixUnit,
                    fy = (float)(int)(__ldg(qi + 32) - fr.ctr[1]) * kFixUnit,
                    fz = (float)(int)(__ldg(qi + 64) - fr.ctr[2]) * kFixUnit;
        const double xi = pos[i], yi = pos[n + i], zi = pos[2 * n + i];
        double ax = 0.0, ay = 0.0, az = 0.0;
        uint32_t pairs = 0, steps = 0, rounds = 0, n_empty = 0, n_live = 0;

        for (uint32_t base = 0; base < blocks.y;) {
            int ne = 0;
            for (; base < blocks.y && ne + 32 <= kEntries64; base += 32) {
                const int nl = live_blocks(base + lane, blocks.y, seg, block_box, fr, cell_f, rcull2, live);
                n_live += nl;
                ++rounds;
                n_empty += nl == 0;
                for (int k = 0; k < nl; ++k) {
                    const LiveBlock S = live.at[k];
                    const uint32_t w = S.word, in = live.slots[k];
                    const uint32_t *qj = relq + (size_t)(w & kBlockMask) * 96 + lane;
                    const uint32_t jx = __ldg(qj), jy = __ldg(qj + 32), jz = __ldg(qj + 64);
                    __syncwarp();  // every lane is done with the previous block's coordinates
                    sj[0][lane] = (float)(int)(jx - S.cx) * kFixUnit;
                    sj[1][lane] = (float)(int)(jy - S.cy) * kFixUnit;
                    sj[2][lane] = (float)(int)(jz - S.cz) * kFixUnit;
                    __syncwarp();
                    uint32_t m = 0;  // slots 8 q .. 8 q + 7 against particle pi
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4 X = *(const float4 *)&sj[0][8 * q + 4 * h], Y = *(const float4 *)&sj[1][8 * q + 4 * h],
                                     Z = *(const float4 *)&sj[2][8 * q + 4 * h];
                        const float xs[4] = {X.x, X.y, X.z, X.w}, ys[4] = {Y.x, Y.y, Y.z, Y.w}, zs[4] = {Z.x, Z.y, Z.z, Z.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float dx = xs[e] - fx, dy = ys[e] - fy, dz = zs[e] - fz;
                            if (dx * dx + dy * dy + dz * dz < rlist2) m |= 1u << (4 * h + e);
                        }
                    }
                    m <<= 8 * q;
                    m |= __shfl_xor_sync(0xffffffffu, m, 8);
                    m |= __shfl_xor_sync(0xffffffffu, m, 16);
                    if (q == 0) mask[ne + k][pi] = valid ? m & in : 0u;
                    if (lane == 0) entry[ne + k] = w;
                }
                ne += nl;
            }
            __syncwarp();
            // this lane's pairs: number q, q + 4, ... of the particle's masks
            int k = 0, skip = q;
            uint32_t m = 0, w = 0;
            for (;;) {
                while (__popc(m) <= skip && k < ne) {
                    skip -= __popc(m);
                    m = mask[k][pi];
                    w = entry[k++];
                }
                const bool have = __popc(m) > skip;
                if (!__any_sync(0xffffffffu, have)) break;
                for (; skip > 0; --skip) m &= m - 1;
                const uint32_t j = have ? (w & kBlockMask) * 32 + (uint32_t)__ffs(m) - 1 : i;
                m &= m - 1;
                skip = have ? 3 : 0;
                double dx = pos[j] - xi, dy = pos[n + j] - yi, dz = pos[2 * n + j] - zi;
                const uint32_t img = have ? seg[w >> 26].image : 0x15u;
                if (__any_sync(0xffffffffu, img != 0x15u)) {  // some pair crosses the boundary
                    const double L = g.box;
                    dx += (img & 3u) == 1u ? 0.0 : ((img & 3u) == 0u ? -L : L);
                    dy += (img >> 2 & 3u) == 1u ? 0.0 : ((img >> 2 & 3u) == 0u ? -L : L);
                    dz += (img >> 4) == 1u ? 0.0 : ((img >> 4) == 0u ? -L : L);
                }
                const double r2 = dx * dx + dy * dy + dz * dz;
                // 0 < r2 < r_c^2 on the bit patterns (non-negative doubles order like integers)
                const long long rb = __double_as_longlong(r2);
                const bool acc = have && rb != 0 && rb < rc2;
                double f = pair_factor64(r2, eps2, kscale, tscale, tab);
                f = acc ? f : 0.0;
                ax = fma(f, dx, ax);
                ay = fma(f, dy, ay);
                az = fma(f, dz, az);
                pairs += acc ? 1u : 0u;
                ++steps;
            }
            __syncwarp();  // the masks are rewritten by the next round
        }
        // the four lanes of a particle, always in the same order
        ax += __shfl_xor_sync(0xffffffffu, ax, 8);
        ay += __shfl_xor_sync(0xffffffffu, ay, 8);
        az += __shfl_xor_sync(0xffffffffu, az, 8);
        ax += __shfl_xor_sync(0xffffffffu, ax, 16);
        ay += __shfl_xor_sync(0xffffffffu, ay, 16);
        az += __shfl_xor_sync(0xffffffffu, az, 16);
        if (valid && q < 3) {  // lane q of a particle writes component q
            const size_t o = (size_t)q * n + i;
            const double a = g.gm * (q == 0 ? ax : (q == 1 ? ay : az));
            const double tot = (acc_in ? acc_in[o] : 0.0) + a;
            acc_out[o] = tot;
            if (kfac != 0.0) mom[o] = __dadd_rn(mom[o], __dmul_rn(kfac, tot));
        }
        st_pairs += __reduce_add_sync(0xffffffffu, pairs);
        st_tested += n_live * kG;
        st_steps += steps;
        st_culled += blocks.y - n_live;
        st_rounds += rounds;
        st_empty += n_empty;
    }
    if (lane == 0) {
        if (st_pairs) {
            atomicAdd(pair_count, st_pairs);
            atomicAdd(pair_count + 1, st_pairs);
        }
        if (st_tested) atomicAdd(pair_count + 3, st_tested);
        if (st_steps) atomicAdd(pair_count + 4, st_steps);
        if (st_culled) atomicAdd(pair_count + 5, st_culled);
        if (st_rounds) atomicAdd(pair_count + 6, st_rounds);
        if (st_empty) atomicAdd(pair_count + 7, st_empty);
    }
}

// ------------------------------------------------------------------ FP32 mode, compacted j lists
// The FP32 kernel.  A work item's up to 32 particles are taken in groups of kG = 16 (8 or 4 when there
// are few, see pair_group; consecutive along the Hilbert order inside the cell, so compact), one group
// at a time per one-warp CTA:
//   1. The neighbour cells form 9 rows of 3 along x, each a contiguous range of sorted slots (two
//      ranges where a row wraps).  The rows' 32-slot blocks are tested 32 at a time, one per lane,
//      against the group's bounding box (block_box, padded by more than its FP32 rounding).
//   2. Lane l of the warp holds slot l of a surviving block and tests that one particle against
//      the group's box; the accepted ones are appended to a list in shared memory (ballot and
//      prefix count), as coordinates relative to the group's centre.  A deep block (all its slots
//      within the cutoff of the whole group: most of a halo's own pairs) goes untested into a list
//      of its own, whose evaluation needs no cutoff (by 10 % of the clustered set's time; near-uniform
//      sets have hardly any).
//   3. Every 32 kChunkBlocks entries the list is evaluated: a lane owns two particles i and takes
//      every (64/kG)-th pair of consecutive entries, two entries at once in packed f32x2
//      arithmetic, so that one 8-byte load per coordinate serves four pair slots.
// Before, 32 particles met every j of the tested blocks, one particle per lane: 37 % of the
// evaluated lane slots held an accepted pair at 200 particles per cell, and half of the
// instructions were tests and votes.  The list holds 47 % accepted slots at kG = 16 (58 % at 8,
// 39 % at 32: the union of the cutoff spheres grows with the group), there are no votes between
// pairs, and a test sequence serves 32 candidates of the whole group.  Measured at 128^3 (one
// evaluation, before / after): near-uniform 5.21 / 3.44 ms, clustered 13.0 / 10.1 ms.
// What bounds it now: of 86 cycles per 32 accepted pairs and scheduler, 61 are the evaluation
// (29 per 32 slots; two FP32 operations with three distinct registers already take three cycles
// of register bandwidth, and a mix of 16 packed operations, 2 rsqrt and 2 ex2 alone runs
// at 20.5), 19 the candidate tests and 6 the set-up of groups.  16 particles per group
// and 18 CTAs per SM: 8, 32 and 16, 20, 24 are within 6 % or slower on both sets.  Two lists of 16 (or
// four of 8) filled by one pass over the candidates save a third of the tests but cost as much in
// registers and reloads (3.18 and 4.8 ms, against 3.06 without the decisions at the cutoff).
//
// Coordinates are 32-bit fixed point, 2^-29 of a chaining cell, modulo 8 cells (relq): differences
// of particles in neighbouring cells, periodic images included, are exact integers, and only the
// difference from the group's centre is rounded to FP32 and scaled (PairFactor).
//
// A pair at r = 0 (the particle itself, or a coincident one) gets a finite factor (r^2 starts at
// kTinyQ when there is no softening) and contributes exactly f * 0.  Only the row of the own cell
// can hold such pairs; there (kOwn) a pair counts only if one of its differences is non-zero.

constexpr int kFlushTerms = 80;         // FP32 terms per partial sum before it joins the FP64 sum
constexpr float kTinyQ = 1e-24f;        // far below the smallest non-zero scaled r^2
constexpr float kFarQ = 1e6f;           // scaled coordinate of a padding entry: outside every cutoff

struct PairConstQ {
    f2 c[5];
    f2 na, ab, e2, tiny;
};

// The factor g(r/r_s) (r^2 + eps^2)^-3/2 of both halves of w (see PairFactor and fit_pair_factor).
// The MUFU pipe takes 8 cycles per warp for a reciprocal or a square root, so that the former
// rsqrt, rcp and sqrt per pair cost as much as 24 FP32 operations; here it is one rsqrt and one
// ex2.  kAdditive (softening small against r_s): 17 FP32 operations per pair with the distance
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
        const f2 s2 = f2_mul(rw, rw), q = f2_fma(k.c[4], s2, f2_fma(k.na, t, f2_add(rw, k.ab)));
        return f2_fma(p, t, f2_fma(q, s2, k.c[0]));
    }
    p = f2_fma(p, t, k.c[0]);
    float sl, sh;
    f2_unpack(f2_add(w, k.e2), sl, sh);
    const f2 s = f2_pack(rsqrt_approx(sl), rsqrt_approx(sh));
    const f2 m = f2_fma(w, p, f2_fma(k.na, t, k.ab));
    const f2 gv = f2_fma(f2_mul(w, rw), m, f2_pack(1.0f, 1.0f));
    return f2_mul(f2_mul(gv, s), f2_mul(s, s));
}

// kAdditive: the form of the pair factor; kG: particles of a group
template <bool kBatched, bool kAdditive, int kChunkBlocks, int kG>
__global__ void __launch_bounds__(32, P3M_PAIR_CTAS)
    k_pairs_list(PairArgs a0, const PairArgs *__restrict__ descs, const uint32_t *__restrict__ order,
                 const uint32_t *__restrict__ n_work_ptr, uint32_t *__restrict__ cursor)
{
    constexpr int kArgWords = sizeof(PairArgs) / 8;
    static_assert(sizeof(PairArgs) % 8 == 0, "PairArgs is copied in 8-byte words");
    constexpr int kChunk = 32 * kChunkBlocks, kCap = kChunk + 32;
    constexpr int kPairsI = kG / 2;              // lanes that share one list entry
    constexpr int kStride = 2 * (32 / kPairsI);  // list entries per warp step
    constexpr int kSub = P3M_PAIR_TI / kG;
    constexpr int kFlushChunks = kFlushTerms * kStride / kChunk < 1 ? 1 : kFlushTerms * kStride / kChunk;
    static_assert(kChunk % kStride == 0, "whole steps per chunk");
    __shared__ __align__(16) float list[3][kCap];
    __shared__ uint32_t slot[kCap];  // the sorted slot of each list entry
    __shared__ __align__(16) float deep[3][kChunk];  // entries within the cutoff of the whole group
    __shared__ double sum[6][32];  // per lane: x, y, z of its first particle, then of its second
    __shared__ PairSeg seg[kPairSegs];
    __shared__ LiveBlocks live;
    __shared__ unsigned long long stat[7];  // pairs, tested, listed, culled, batches, empty batches, deep
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
        if (lane < 7) stat[lane] = 0ull;
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
        if (lane < 7 && stat[lane]) {
            atomicAdd(A.pair_count + (lane == 6 ? 2 : lane + (lane ? 2 : 1)), stat[lane]);
            if (lane == 0) atomicAdd(A.pair_count, stat[0]);
        }
    };
    if (!kBatched) load_args(&a0);

    for (;;) {
        uint32_t unit = 0;
        if (lane == 0) unit = atomicAdd(cursor, 1u);
        unit = __shfl_sync(0xffffffffu, unit, 0);
        if (unit >= n_units) break;
        uint32_t item = kBatched ? order[unit / kSub] : unit / kSub;
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

        const GroupFrame fr = group_frame<kG>(A.relq, first, cend, cx, cy, cz, A.fac.lambda, A.fac.cell);
        const uint2 blocks = group_ranges(seg, A.cell_start, g, cx, cy, cz, fr, A.fac.cell);
        const float hx = fr.half[0], hy = fr.half[1], hz = fr.half[2];
#pragma unroll
        for (int q = 0; q < 6; ++q) sum[q][lane] = 0.0;

        // the lane's two particles, relative to the centre and negated
        const float lambda = A.fac.lambda;
        f2 nx[2], ny[2], nz[2], px[2], py[2], pz[2];
        uint32_t cnt[2] = {0u, 0u};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const uint32_t i = min(first + ip + u * kPairsI, cend - 1);
            const uint32_t *q = fix_coords(A.relq, i);
            const float x = (float)(int)(__ldg(q) - fr.ctr[0]) * -lambda,
                        y = (float)(int)(__ldg(q + 32) - fr.ctr[1]) * -lambda,
                        z = (float)(int)(__ldg(q + 64) - fr.ctr[2]) * -lambda;
            nx[u] = f2_pack(x, x);
            ny[u] = f2_pack(y, y);
            nz[u] = f2_pack(z, z);
            px[u] = py[u] = pz[u] = f2_pack(0.0f, 0.0f);
        }
        const float rlist2 = A.fac.rlist2;
        const float cut_m = kBatched ? A.fac.cut_m : a0.fac.cut_m, cut_b = kBatched ? A.fac.cut_b : a0.fac.cut_b;
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
        // The pairs of a list in the cutoff's band: their terms are made whole or taken back, and so are
        // their parts of the sums of cut_part (total).
        auto settle = [&](auto additive, int count, float *total) {
            constexpr bool kAdd = decltype(additive)::value;
#pragma unroll 1
            for (int k = 0; k < 2 * count; k += kStride) {
                const int p = (k < count ? k : k - count + 1) + 2 * js;  // the first, then the second halves
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const float dx = list[0][p] + nx[u].x, dy = list[1][p] + ny[u].x, dz = list[2][p] + nz[u].x;
                    const float w = fmaf(dz, dz, fmaf(dy, dy, fmaf(dx, dx, kAdd ? kc.e2.x : kTinyQ)));
                    const float part = cut_part(w, cut_m, cut_b);
                    if (part == rintf(part)) continue;
                    const uint32_t i = min(first + ip + u * kPairsI, cend - 1);
                    const float t = (cut_inside<false>(A.relq, {A.rel, A.keys}, g, i, slot[p], dx, dy, dz, A.fac) ? 1.0f : 0.0f) - part;
                    const float f = t * pair_factor_q<kAdd>(f2_pack(w, w), kc).x;
                    px[u].x = fmaf(f, dx, px[u].x);
                    py[u].x = fmaf(f, dy, py[u].x);
                    pz[u].x = fmaf(f, dz, pz[u].x);
                    total[u] += t;
                }
            }
        };
        // list entries [0, count), count a multiple of kStride
        auto eval_form = [&](auto additive, auto own, int count) {
            constexpr bool kAdd = decltype(additive)::value;
            const f2 w0 = kAdd ? kc.e2 : kc.tiny;
            const float *lx = &list[0][2 * js], *ly = &list[1][2 * js], *lz = &list[2][2 * js];
            f2 Xn = *(const f2 *)lx, Yn = *(const f2 *)ly, Zn = *(const f2 *)lz;
            f2 hits[2] = {f2_pack(0.0f, 0.0f), f2_pack(0.0f, 0.0f)};
#pragma unroll 2
            for (int k = 0; k < count; k += kStride) {
                const f2 X = Xn, Y = Yn, Z = Zn;
                const int kn = k + kStride < count ? k + kStride : 0;
                Xn = *(const f2 *)(lx + kn), Yn = *(const f2 *)(ly + kn), Zn = *(const f2 *)(lz + kn);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const f2 dx = f2_add(X, nx[u]), dy = f2_add(Y, ny[u]), dz = f2_add(Z, nz[u]);
                    const f2 w = f2_fma(dz, dz, f2_fma(dy, dy, f2_fma(dx, dx, w0)));
                    f2 f = pair_factor_q<kAdd>(w, kc);
                    const f2 in = f2_pack(cut_part(w.x, cut_m, cut_b), cut_part(w.y, cut_m, cut_b));
                    f = f2_mul(f, in);
                    px[u] = f2_fma(f, dx, px[u]);
                    py[u] = f2_fma(f, dy, py[u]);
                    pz[u] = f2_fma(f, dz, pz[u]);
                    if (decltype(own)::value) {
                        const bool nl = (__float_as_uint(dx.x) | __float_as_uint(dy.x) | __float_as_uint(dz.x)) != 0u;
                        const bool nh = (__float_as_uint(dx.y) | __float_as_uint(dy.y) | __float_as_uint(dz.y)) != 0u;
                        hits[u] = f2_add(hits[u], f2_pack(nl ? in.x : 0.0f, nh ? in.y : 0.0f));
                    } else {
                        hits[u] = f2_add(hits[u], in);
                    }
                }
            }
            // a sum with a fraction holds a pair in the band
            float total[2] = {hits[0].x + hits[0].y, hits[1].x + hits[1].y};
            const bool near = total[0] != rintf(total[0]) || total[1] != rintf(total[1]);
            if (__any_sync(0xffffffffu, near)) settle(additive, count, total);
            cnt[0] += __float2uint_rn(total[0]);
            cnt[1] += __float2uint_rn(total[1]);
        };
        // the same for the deep entries [0, count): no pair is cut off, only the own row's r = 0 do not count
        auto deep_form = [&](auto additive, auto own, int count) {
            constexpr bool kAdd = decltype(additive)::value;
            const f2 w0 = kAdd ? kc.e2 : kc.tiny;
            const float *lx = &deep[0][2 * js], *ly = &deep[1][2 * js], *lz = &deep[2][2 * js];
            f2 Xn = *(const f2 *)lx, Yn = *(const f2 *)ly, Zn = *(const f2 *)lz;
#pragma unroll 2
            for (int k = 0; k < count; k += kStride) {
                const f2 X = Xn, Y = Yn, Z = Zn;
                const int kn = k + kStride < count ? k + kStride : 0;
                Xn = *(const f2 *)(lx + kn), Yn = *(const f2 *)(ly + kn), Zn = *(const f2 *)(lz + kn);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const f2 dx = f2_add(X, nx[u]), dy = f2_add(Y, ny[u]), dz = f2_add(Z, nz[u]);
                    const f2 w = f2_fma(dz, dz, f2_fma(dy, dy, f2_fma(dx, dx, w0)));
                    const f2 f = pair_factor_q<kAdd>(w, kc);
                    px[u] = f2_fma(f, dx, px[u]);
                    py[u] = f2_fma(f, dy, py[u]);
                    pz[u] = f2_fma(f, dz, pz[u]);
                    if (decltype(own)::value) {
                        if ((__float_as_uint(dx.x) | __float_as_uint(dy.x) | __float_as_uint(dz.x)) != 0u) ++cnt[u];
                        if ((__float_as_uint(dx.y) | __float_as_uint(dy.y) | __float_as_uint(dz.y)) != 0u) ++cnt[u];
                    }
                }
            }
            if (!decltype(own)::value) {
                cnt[0] += 2 * count / kStride;
                cnt[1] += 2 * count / kStride;
            }
        };
        auto eval = [&](auto own, int count) { eval_form(std::bool_constant<kAdditive>{}, own, count); };
        auto eval_deep = [&](auto own, int count) { deep_form(std::bool_constant<kAdditive>{}, own, count); };

        uint32_t n_list = 0, n_live = 0, n_chunks = 0;
        int fill = 0, fill_deep = 0;
        // the blocks [t0, t1) of the ranges in sequence
        auto walk = [&](auto own, uint32_t t0, uint32_t t1) {
            for (uint32_t base = t0; base < t1; base += 32) {
                const int nl = live_blocks(base + lane, t1, seg, A.block_box, fr, A.fac.length, A.rcull2, live, A.rin2);
                n_live += nl;
                if (nl == 0 && lane == 0) ++stat[5];
                // the next block's coordinates are loaded while the current one is tested
                uint32_t xn = 0, yn = 0, zn = 0;
                auto fetch = [&](int k) {
                    const uint32_t *q = relq + (size_t)(live.at[k].word & kBlockMask) * 96;
                    xn = __ldg(q);
                    yn = __ldg(q + 32);
                    zn = __ldg(q + 64);
                };
                if (nl) fetch(0);
#pragma unroll 1
                for (int k = 0; k < nl; ++k) {
                    const LiveBlock S = live.at[k];
                    const float x = (float)(int)(xn - S.cx) * lambda, y = (float)(int)(yn - S.cy) * lambda,
                                z = (float)(int)(zn - S.cz) * lambda;
                    const bool mine = live.slots[k] >> lane & 1u;
                    if (k + 1 < nl) fetch(k + 1);
                    if (S.word & kDeepBlock) {
                        deep[0][fill_deep + lane] = x;
                        deep[1][fill_deep + lane] = y;
                        deep[2][fill_deep + lane] = z;
                        fill_deep += 32;
                        if (fill_deep == kChunk) {
                            __syncwarp();
                            eval_deep(own, kChunk);
                            __syncwarp();
                            fill_deep = 0;
                            if (lane == 0) stat[6] += kChunk / 32 * kG;
                            if (++n_chunks % kFlushChunks == 0) flush();
                        }
                        continue;
                    }
                    const float ex = fmaxf(fabsf(x) - hx, 0.0f), ey = fmaxf(fabsf(y) - hy, 0.0f),
                                ez = fmaxf(fabsf(z) - hz, 0.0f);
                    const bool in = mine && ex * ex + ey * ey + ez * ez < rlist2;
                    const uint32_t mm = __ballot_sync(0xffffffffu, in);
                    if (in) {
                        const int p = fill + __popc(mm & lt);
                        list[0][p] = x;
                        list[1][p] = y;
                        list[2][p] = z;
                        slot[p] = (S.word & kBlockMask) << 5 | lane;
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
                            slot[lane] = slot[kChunk + lane];
                        }
                        n_list += kChunk;
                        if (++n_chunks % kFlushChunks == 0) flush();
                    }
                }
            }
            // the rest of the list, padded to whole steps with far entries
            const int count = (fill + kStride - 1) / kStride * kStride;
            if (lane < count - fill) list[0][fill + lane] = list[1][fill + lane] = list[2][fill + lane] = kFarQ;
            __syncwarp();
            eval(own, count);
            if (fill_deep) eval_deep(own, fill_deep);
            __syncwarp();
            flush();
            n_list += fill;
            if (fill_deep && lane == 0) stat[6] += fill_deep / 32 * kG;
            fill = fill_deep = 0;
        };
        walk(std::true_type{}, 0u, blocks.x);
        walk(std::false_type{}, blocks.x, blocks.y);
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
            stat[1] += n_live * kG;              // j's of the blocks near the group (deep ones too), in slots of 32
            stat[2] += (n_list * kG + 16) / 32;  // list entries evaluated after a test, the same
            stat[3] += blocks.y - n_live;
            stat[4] += (blocks.x + 31) / 32 + (blocks.y - blocks.x + 31) / 32;
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
    // culling radius: r_c widened by more than the FP32 rounding of absolute coordinates up to the
    // box size; candidate radius (in cell sides): by more than the FP32 rounding of differences of up
    // to two cells
    const double rcull = c->g.r_c * (1.0 + 1e-4) + c->g.box * 1e-6, rlist = c->g.r_c / c->g.cs + 2e-6;
    c->launches += 1;
    k_pairs64<<<grid, 32, 0, c->stream>>>(c->relq, c->pos, c->block_box, c->cell_start, c->work,
                                          c->n_work, c->g, c->split_tab,
                                          (float)(rcull * rcull), (float)(rlist * rlist), acc_in, acc_out,
                                          c->mom, kfac, kfac_dev, c->counters, c->pair_count);
    return cudaGetLastError();
}

// The FP32 kernel for one context or (batched) several.
template <bool kBatched, bool kAdditive, int kChunkBlocks, int kG>
cudaError_t launch_list(const PairArgs &a, const PairArgs *descs, const uint32_t *order,
                        const uint32_t *n_work, uint32_t *cursor, int num_sms, cudaStream_t s)
{
    int per_sm = 0;
    auto kern = k_pairs_list<kBatched, kAdditive, kChunkBlocks, kG>;
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
    const bool add = c->pair_factor.additive != 0;
    const int group = pair_group(c);
    auto launch = group == 4   ? (add ? launch_list<false, true, kLongChunk, 4> : launch_list<false, false, kLongChunk, 4>)
                  : group == 8 ? (add ? launch_list<false, true, kLongChunk, 8> : launch_list<false, false, kLongChunk, 8>)
                  : c->tile_blocks == kShortChunk
                      ? (add ? launch_list<false, true, kShortChunk, 16> : launch_list<false, false, kShortChunk, 16>)
                      : (add ? launch_list<false, true, kLongChunk, 16> : launch_list<false, false, kLongChunk, 16>);
    return launch(a, nullptr, nullptr, c->n_work, c->counters, c->num_sms, c->stream);
}

__global__ void k_store_pair_args(PairArgs *dst, PairArgs a) { *dst = a; }

__global__ void k_ens_gather(uint32_t slot, const uint32_t *__restrict__ key,
                             size_t n, uint32_t *__restrict__ gk, uint32_t *__restrict__ gv)
{
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n;
         k += (size_t)gridDim.x * blockDim.x) {
        gk[k] = key[k];
        gv[k] = (slot << 24) | ((uint32_t)k & 0xFFFFFFu);
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
    a.rel = (const float4 *)c->rel;
    a.keys = c->keys;
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
    const double rin = c->g.r_c * (1.0 - 1e-4) - c->g.box * 1e-6;
    a.rin2 = rin > 0.0 ? (float)(rin * rin) : -1.0f;

    return a;
}

cudaError_t launch_pairs_batched(const PairArgs *descs, const uint32_t *order,
                                 const uint32_t *n_total, uint32_t *cursor, int group, int num_sms,
                                 cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(cursor, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    PairArgs unused;
    memset(&unused, 0, sizeof(unused));
    auto launch = group == 16  ? launch_list<true, true, kLongChunk, 16>
                  : group == 8 ? launch_list<true, true, kLongChunk, 8>
                               : launch_list<true, true, kLongChunk, 4>;
    return launch(unused, descs, order, n_total, cursor, num_sms, s);
}

cudaError_t launch_store_pair_args(PairArgs *dst, const PairArgs &a, cudaStream_t s)
{
    k_store_pair_args<<<1, 1, 0, s>>>(dst, a);
    return cudaGetLastError();
}

cudaError_t launch_ens_gather(int slot, const uint32_t *key, size_t n, uint32_t *gkey, uint32_t *gval, cudaStream_t s)
{
    const size_t blocks = (n + 255) / 256;
    k_ens_gather<<<(unsigned)(blocks < 1 ? 1 : (blocks > 1024 ? 1024 : blocks)), 256, 0, s>>>(
        (uint32_t)slot, key, n, gkey, gval);
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
