// The walk over the neighbourhood of a group of particles that the pair kernels share.  A group is up
// to 32 consecutive particles of one chaining cell, handled by one warp.  Its neighbour cells form 9
// rows of 3 along x, each a contiguous range of sorted slots (two ranges where a row wraps); the
// ranges' 32-slot blocks are tested 32 at a time, one per lane, against the group's bounding box.
#pragma once

#include <cuda_runtime.h>

#include "p3m_internal.cuh"

namespace {

constexpr int kPairSegs = 18;  // 9 rows of neighbour cells, each at most two ranges

// The group's bounding box around an integer centre (fixed-point coordinates, kFixBits): centre,
// half extents (scaled by lambda, rounded up), and the centre in absolute FP32 coordinates.
struct GroupFrame {
    uint32_t ctr[3];
    float half[3], actr[3];
};

// One range of neighbour slots of a group: its slots, the group's centre in the range's periodic
// image (fixed point, and absolute FP32 for the block boxes), the number of blocks before it and
// the image as 3 x 2 bits (image index + 1).
struct __align__(16) PairSeg {
    uint32_t start, end, cx, cy;
    uint32_t cz, first_block;
    float ax, ay;
    float az;
    uint32_t image, pad[2];
};

__device__ __forceinline__ const uint32_t *fix_coords(const uint32_t *relq, uint32_t i)
{
    return relq + (size_t)(i >> 5) * 96 + (i & 31);
}

// Frame of the particles [first, min(first + kG, cend)) of cell (cx, cy, cz).
template <int kG>
__device__ __forceinline__ GroupFrame group_frame(const uint32_t *relq, uint32_t first, uint32_t cend,
                                                  int cx, int cy, int cz, float lambda, float cell)
{
    GroupFrame f;
    const int lane = threadIdx.x & 31;
    const uint32_t *q = fix_coords(relq, min(first + min(lane, kG - 1), cend - 1));
    const int c3[3] = {cx, cy, cz};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const uint32_t x = __ldg(q + 32 * d), x0 = __shfl_sync(0xffffffffu, x, 0);
        const int lo = __reduce_min_sync(0xffffffffu, (int)(x - x0));
        const int hi = __reduce_max_sync(0xffffffffu, (int)(x - x0));
        const int mid = lo + ((hi - lo) >> 1);
        f.ctr[d] = x0 + (uint32_t)mid;
        f.half[d] = (float)(max(hi - mid, mid - lo)) * (1.0f + 0x1p-20f) * lambda;
        // cell index and offset inside the cell, in cell sides
        f.actr[d] = ((float)c3[d] + (float)(int)(f.ctr[d] - ((uint32_t)c3[d] << kFixBits)) * kFixUnit) * cell;
    }
    return f;
}

// Fills seg (the own row's two ranges first); returns the number of blocks of the own row and of all.
__device__ __forceinline__ uint2 group_ranges(PairSeg *seg, const uint32_t *cell_start, const P3MGeom &g,
                                              int cx, int cy, int cz, const GroupFrame &f, float cell)
{
    const int lane = threadIdx.x & 31, nc = g.n_c;
    __syncwarp();  // the previous group is done with seg
    uint32_t blocks = 0;
    if (lane < kPairSegs) {
        const int row = ((lane >> 1) + 4) % 9;  // the own row (4) comes first
        const int uy = cy + row % 3 - 1, uz = cz + row / 3 - 1;
        const int iy = uy < 0 ? -1 : (uy >= nc ? 1 : 0), iz = uz < 0 ? -1 : (uz >= nc ? 1 : 0);
        int x0 = max(cx - 1, 0), x1 = min(cx + 1, nc - 1), ix = 0;
        if (lane & 1) {  // the wrapped end of the row, if any
            ix = cx == 0 ? -1 : (cx == nc - 1 ? 1 : 0);
            x0 = x1 = cx == 0 ? nc - 1 : 0;
        }
        const uint32_t base = ((uint32_t)(uz - iz * nc) * nc + (uint32_t)(uy - iy * nc)) * nc;
        uint32_t s = cell_start[base + x0], e = cell_start[base + x1 + 1];
        if (!p3m_in_bounds(s <= e && e <= (uint32_t)g.n, g.flags)) e = s;
        if ((lane & 1) && ix == 0) e = s;
        PairSeg q;
        q.start = s;
        q.end = e;
        const uint32_t box = (uint32_t)nc << kFixBits;  // the box side modulo 2^32
        q.cx = f.ctr[0] - (uint32_t)ix * box;
        q.cy = f.ctr[1] - (uint32_t)iy * box;
        q.cz = f.ctr[2] - (uint32_t)iz * box;
        q.ax = f.actr[0] - (float)(ix * nc) * cell;
        q.ay = f.actr[1] - (float)(iy * nc) * cell;
        q.az = f.actr[2] - (float)(iz * nc) * cell;
        q.image = (uint32_t)(ix + 1) | (uint32_t)(iy + 1) << 2 | (uint32_t)(iz + 1) << 4;
        q.pad[0] = q.pad[1] = 0;
        const uint32_t mine = e > s ? ((e - 1) >> 5) - (s >> 5) + 1 : 0;
        blocks = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync((1u << kPairSegs) - 1u, blocks, o);
            if (lane >= o) blocks += y;
        }
        q.first_block = blocks - mine;
        seg[lane] = q;
    }
    __syncwarp();
    return make_uint2(__shfl_sync(0xffffffffu, blocks, 1), __shfl_sync(0xffffffffu, blocks, kPairSegs - 1));
}

// A surviving block: (range << 26) | block, the group's centre in its image, and its slots that belong
// to the range.  kDeepBlock in the word: all 32 slots do, and all are within the cutoff of all of the group.
struct __align__(16) LiveBlock {
    uint32_t word, cx, cy, cz;
};
struct LiveBlocks {
    LiveBlock at[32];
    uint32_t slots[32];
};
constexpr uint32_t kBlockMask = 0x3FFFFFFu, kDeepBlock = 0x80000000u;

// Tests block t of the ranges in sequence (t >= t1: none) against the group's box; the survivors of
// the warp's 32 blocks go to live[0 ..] in order.  Returns their number.
// rin2: the squared cutoff less the same margins (no deep blocks if negative).
// length: one scaled length (as in f.half); rcull2: the squared cutoff, padded by more than the FP32
// rounding of absolute coordinates.
__device__ __forceinline__ int live_blocks(uint32_t t, uint32_t t1, const PairSeg *seg,
                                           const float4 *block_box, const GroupFrame &f, float length,
                                           float rcull2, LiveBlocks &live, float rin2 = -1.0f)
{
    const int lane = threadIdx.x & 31;
    bool keep = false;
    LiveBlock q = {0u, 0u, 0u, 0u};
    uint32_t slots = 0;
    if (t < t1) {
        int s = 0;  // the last range that starts at or before block t
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            if (s + o < kPairSegs && seg[s + o].first_block <= t) s += o;
        const PairSeg &S = seg[s];
        const uint32_t b = (S.start >> 5) + (t - S.first_block);
        const float4 lo = __ldg(block_box + 2 * (size_t)b), hi = __ldg(block_box + 2 * (size_t)b + 1);
        const float ex = fmaxf(fmaxf(lo.x - S.ax, S.ax - hi.x) - f.half[0] * length, 0.0f);
        const float ey = fmaxf(fmaxf(lo.y - S.ay, S.ay - hi.y) - f.half[1] * length, 0.0f);
        const float ez = fmaxf(fmaxf(lo.z - S.az, S.az - hi.z) - f.half[2] * length, 0.0f);
        keep = ex * ex + ey * ey + ez * ez < rcull2;
        const uint32_t j0 = max(b * 32, S.start) - b * 32, j1 = min(S.end - b * 32, 32u);
        slots = (0xffffffffu << j0) & (0xffffffffu >> (32 - j1));  // (0 <= j0 < j1 <= 32)
        q = {((uint32_t)s << 26) | b, S.cx, S.cy, S.cz};
        const float mx = fmaxf(hi.x - S.ax, S.ax - lo.x) + f.half[0] * length,
                    my = fmaxf(hi.y - S.ay, S.ay - lo.y) + f.half[1] * length,
                    mz = fmaxf(hi.z - S.az, S.az - lo.z) + f.half[2] * length;
        if (slots == 0xffffffffu && mx * mx + my * my + mz * mz < rin2) q.word |= kDeepBlock;
    }
    const uint32_t m = __ballot_sync(0xffffffffu, keep);
    __syncwarp();  // every lane is done with the previous survivors
    if (keep) {
        const int k = __popc(m & ((1u << lane) - 1u));
        live.at[k] = q;
        live.slots[k] = slots;
    }
    __syncwarp();
    return __popc(m);
}

// ------------------------------------------------------------------ the cutoff
// Which pairs interact must not depend on a kernel's layout: the force jumps at the cutoff, and one pair on
// the other side moves a component of a nearly uniform set by up to 3e-3 of the rms force.  The FP32 mode
// decides r < r_c by the FP32 r^2 of the cell-relative coordinates, of x_j and of x_i shifted into j's
// cell (cut_inside), which is within 8e-8 (rms) of the exact one at the cutoff: about one pair in 10^7
// falls on the other side of it.  A set with fewer particles than chaining cells, where a pair may be all of a
// particle's force, is decided by the fixed-point coordinates instead (PairFactor::fix_rc2).
// The lists' own r^2 is rounded differently, so the kernels evaluate with a factor that is 1 inside, 0
// outside and a fraction within kCutBand, sum it per lane (it also counts the pairs), and where a sum has a
// fraction (one list of 160 in 600) look at the list again and decide its pairs in the band.  (Two fractions
// of one lane whose sum is a whole number to 2^-18 would hide each other.)  Two clamped FMAs, a product and a sum
// per two pairs take 4 % of the force kernel's time; compares, selects and counts beside a minimum of
// |w - rc2| took 9 %.

// 1 inside the cutoff, 0 outside
__device__ __forceinline__ float cut_part(float w, float cut_m, float cut_b)
{
    return __saturatef(fmaf(w, cut_m, cut_b));
}

// r < r_c by FP32, i and j in neighbouring chaining cells (n_c >= 3: the two cells give the periodic image).
__device__ __forceinline__ bool cut_inside_fp32(const float4 *rel, const uint32_t *keys, int sub_bits, int nc, double cs,
                                                double box, float rc2, uint32_t i, uint32_t j)
{
    uint32_t ci = keys[i] >> (3 * sub_bits), cj = keys[j] >> (3 * sub_bits);
    const float4 a = rel[i], b = rel[j];
    const float xi[3] = {a.x, a.y, a.z}, xj[3] = {b.x, b.y, b.z};
    float r2 = 1e-20f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int c = (int)(ci % (uint32_t)nc), w = (int)(cj % (uint32_t)nc);
        ci /= (uint32_t)nc;
        cj /= (uint32_t)nc;
        const double image = w - c > 1 ? -box : (w - c < -1 ? box : 0.0);
        // the two cells' origins differ by s, an FP32 value and its FP32 residual
        const double s = ((double)w * cs + image) - (double)c * cs;
        const float hi = (float)s, lo = (float)(s - (double)hi);
        const float x = xj[d] - ((xi[d] - hi) - lo);
        r2 = fmaf(x, x, r2);
    }
    return r2 < rc2;
}

// (A call in the force kernel, one in thousands of pairs: its registers are at their limit.  The VJP kernel
// has some to spare and is 1.5 % faster with the function inlined.)
__device__ __noinline__ bool cut_inside_fp32_call(const float4 *rel, const uint32_t *keys, int sub_bits, int nc, double cs,
                                                  double box, float rc2, uint32_t i, uint32_t j)
{
    return cut_inside_fp32(rel, keys, sub_bits, nc, cs, box, rc2, i, j);
}

// What the decision on a pair in the band reads beside the fixed-point coordinates.
struct CutState {
    const float4 *rel;     // relative to the cells' origins, sorted order
    const uint32_t *keys;  // sorted
};

// Whether i and j, whose scaled FP32 difference is (dx, dy, dz), are closer than the cutoff.
template <bool kInline>
__device__ __forceinline__ bool cut_inside(const uint32_t *relq, const CutState &st, const P3MGeom &g, uint32_t i,
                                           uint32_t j, float dx, float dy, float dz, const PairFactor &f)
{
    if (f.fix_rc2 == 0)
        return (kInline ? cut_inside_fp32 : cut_inside_fp32_call)(st.rel, st.keys, g.sub_bits, g.n_c, g.cs, g.box, f.fp32_rc2, i, j);
    const uint32_t *qi = fix_coords(relq, i), *qj = fix_coords(relq, j);
    const float d3[3] = {dx, dy, dz};
    long long r2 = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        // the difference of the images: known up to whole cells from the coordinates, which cell from FP32
        constexpr uint32_t kCell = 1u << kFixBits;
        const uint32_t e = __ldg(qj + 32 * d) - __ldg(qi + 32 * d), near = (uint32_t)(int)(d3[d] / f.lambda);
        const long long x = (int)(e + ((near - e + kCell / 2) & ~(kCell - 1u)));
        r2 += x * x;
    }
    return r2 < f.fix_rc2;
}

}  // namespace
