// Chaining-cell keys, stable LSD radix sort, particle permutation, cell ranges and the
// pair work list.
//
// Key of a particle (the chaining-mesh binning of P3M; the guide only fixes the cutoff that
// sets the cell size, Ch. Parameters "P3M_cutoff"): with n_f = n_c 2^b fine cells per side,
//   f_d = min(trunc(x_d * (n_f / L)), n_f - 1)   (one correctly rounded FP64 multiply)
//   cell = (c_z n_c + c_y) n_c + c_x,  c_d = f_d >> b
//   key  = (cell << 3b) | Hilbert(f_x mod 2^b, f_y mod 2^b, f_z mod 2^b)
// (Hilbert: the index along the 3-D Hilbert curve of order b, after Skilling, "Programming the
// Hilbert curve", AIP Conf. Proc. 707, 2004; consecutive indices are face neighbours, so runs of
// consecutive particles are more compact than along a Morton order)
// Particles are ordered by key, ties by their current slot (a stable sort), so the order is
// reproducible bit for bit.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <mutex>
#include <type_traits>

#include "p3m_internal.cuh"
#include "state.cuh"
#include "work_list.h"

namespace {

constexpr int kThreads = 256;
constexpr int kItems = P3M_SORT_TILE / kThreads;  // 16
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;

// (not inlined: the compiler would otherwise run the FP64 product for every particle)
__device__ __noinline__ uint32_t fine_index(double x, double inv, int nf)
{
    int f = (int)__dmul_rn(x, inv);  // x >= 0: truncation is floor
    return (uint32_t)min(f, nf - 1);
}

// The same index without FP64 arithmetic in almost every case.  x_f = x truncated to its
// leading 24 significant bits (bit operations), inv_f = inv rounded to FP32: the FP32 product
// p = x_f inv_f is within 2^-22 x inv < 2^-22 n_f of x inv, and the correctly rounded FP64
// product within 2^-53 n_f of it.  So when p lies more than tol = 2^-21 n_f from every
// integer, floor(p) is floor of the FP64 product; otherwise the FP64 product decides.
__device__ __forceinline__ uint32_t fine_index_fast(double x, double inv, float inv_f, float tol, int nf)
{
    const long long xb = __double_as_longlong(x);
    const int e = (int)((xb >> 52) & 0x7FF) - 1023 + 127;  // x >= 0: no sign bit
    const float xf = e >= 1 ? __int_as_float((e << 23) | (int)((xb >> 29) & 0x7FFFFF)) : 0.0f;
    const float p = xf * inv_f;
    // floor(p) in the low bits of p + 2^23 rounded towards zero (0 <= p < 2^23)
    const float t = __fadd_rz(p, 8388608.0f), fr = p - (t - 8388608.0f);
    if (fr > tol && fr < 1.0f - tol) return (uint32_t)min(__float_as_int(t) & 0x7FFFFF, nf - 1);
    return fine_index(x, inv, nf);
}

// kBits: sub_bits at compile time, or -1 (any)
template <int kBits>
__device__ __forceinline__ uint32_t make_key(uint32_t fx, uint32_t fy, uint32_t fz,
                                             const P3MGeom &g)
{
    const int b = kBits >= 0 ? kBits : g.sub_bits;
    const uint32_t cell = ((fz >> b) * (uint32_t)g.n_c + (fy >> b)) * (uint32_t)g.n_c + (fx >> b);
    const uint32_t m = (1u << b) - 1u;
    uint32_t x[3] = {fx & m, fy & m, fz & m}, code = 0;
    if (b > 0) {
        const uint32_t top = 1u << (b - 1);
#pragma unroll
        for (uint32_t q = top; q > 1; q >>= 1) {  // undo the excess rotations and reflections
            const uint32_t low = q - 1;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                if (x[i] & q) {
                    x[0] ^= low;
                } else {
                    const uint32_t t = (x[0] ^ x[i]) & low;
                    x[0] ^= t;
                    x[i] ^= t;
                }
            }
        }
        x[1] ^= x[0];  // Gray encode
        x[2] ^= x[1];
        uint32_t t = 0;
#pragma unroll
        for (uint32_t q = top; q > 1; q >>= 1)
            if (x[2] & q) t ^= q - 1;
        for (int i = 0; i < 3; ++i) x[i] ^= t;
#pragma unroll
        for (int level = b - 1; level >= 0; --level)
#pragma unroll
            for (int i = 0; i < 3; ++i) code = (code << 1) | ((x[i] >> level) & 1u);
    }
    return (cell << (3 * b)) | code;
}

// hist[d] += 1 of every valid lane.  A warp whose digits agree (the upper digits of a set that is nearly
// sorted) adds once, the others one by one in shared memory.
__device__ __forceinline__ void count_digit(uint32_t *hist, uint32_t d, bool valid, int lane)
{
    const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
    if (__all_sync(0xffffffffu, valid && d == d0)) {
        if (lane == 0) atomicAdd(&hist[d0], 32u);
    } else if (valid) {
        atomicAdd(&hist[d], 1u);
    }
}

// Half kick + drift (optional), periodic wrap, key.  Kick and drift are one FMA each (a single
// rounding): p += (m K) a; x += p (D / m).  With fac_dev the two factors are read from
// fac_dev[0], fac_dev[1] (graph-replayed steps).
// Bound by memory (28 bytes per particle, 124 with the kick) once the FP64 compares are out of the way
// and the Hilbert index is unrolled: 256^3 without a kick 0.381 -> 0.159 ms.  A position that is inside the
// box already is not written again.
// kHist (the sort by look-back follows): hist[p 256 + d] += keys whose digit p is d, p < passes, by shared-memory
// atomics; a kernel of its own took 4 to 5 us of a small set's evaluation.
template <int kBits, bool kKick, bool kHist>
__global__ void __launch_bounds__(256, 6)
    k_kick_drift_keys(double *__restrict__ pos, double *__restrict__ mom, const double *__restrict__ acc,
                      P3MGeom g, double kfac, double dfac, uint32_t *__restrict__ keys,
                      const double *__restrict__ fac_dev, int passes, uint32_t *__restrict__ hist)
{
    __shared__ uint32_t h[kHist ? 4 * kRadix : 1];
    if (kHist) {
        for (int i = threadIdx.x; i < passes * kRadix; i += kThreads) h[i] = 0;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int64_t n = g.n;
    if (kKick && fac_dev) {
        kfac = fac_dev[0];
        dfac = fac_dev[1];
    }
    const float inv_f = (float)g.inv_fine, tol = (float)g.n_fine * 0x1p-21f;
    for (int64_t i0 = blockIdx.x * (int64_t)kThreads; i0 < n; i0 += (int64_t)gridDim.x * kThreads) {
        const int64_t i = i0 + threadIdx.x;
        uint32_t key = 0;
        if (i < n) {
            uint32_t f[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                double x = pos[d * n + i];
                const double x0 = x;
                if (kKick) {
                    const double p = __fma_rn(kfac, acc[d * n + i], mom[d * n + i]);
                    mom[d * n + i] = p;
                    x = __fma_rn(p, dfac, x);
                }
                x = wrap_box(x, g.box);
                if (__double_as_longlong(x) != __double_as_longlong(x0)) pos[d * n + i] = x;
                f[d] = fine_index_fast(x, g.inv_fine, inv_f, tol, g.n_fine);
            }
            key = make_key<kBits>(f[0], f[1], f[2], g);
            p3m_in_bounds((key >> (3 * g.sub_bits)) < (uint32_t)g.n_cells, g.flags);
            keys[i] = key;
        }
        if (kHist)
            for (int p = 0; p < passes; ++p)
                count_digit(h + p * kRadix, (key >> (p * kRadixBits)) & (kRadix - 1), i < n, lane);
    }
    if (kHist) {
        __syncthreads();
        for (int i = threadIdx.x; i < passes * kRadix; i += kThreads)
            if (h[i]) atomicAdd(hist + i, h[i]);
    }
}

// ------------------------------------------------------------------ radix sort, 8-bit digits

// The valid lanes whose digit (bits wide) equals this lane's, from one ballot per bit: about 40
// instructions, where __match_any_sync takes some ten cycles per distinct digit, 300 for random ones.
__device__ __forceinline__ uint32_t match_digit(uint32_t d, bool valid, int bits)
{
    uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int b = 0; b < kRadixBits; ++b) {
        if (b >= bits) break;
        const uint32_t one = d >> b & 1u;
        peers &= ~(__ballot_sync(0xffffffffu, one) ^ (0u - one));
    }
    return peers;
}

// Tile t holds keys [t*4096, (t+1)*4096), visited in 16 rounds of 256 consecutive keys;
// within a round warp w holds keys [w*32, w*32+32).  That visiting order is the input order,
// so ranks assigned round by round, warp by warp, lane by lane make each pass stable.

__global__ void __launch_bounds__(kThreads)
    k_radix_upsweep(const uint32_t *__restrict__ keys, int64_t n, int shift,
                    uint32_t *__restrict__ counts, int n_tiles)
{
    __shared__ uint32_t hist[kRadix];
    const int tid = threadIdx.x, lane = tid & 31;
    hist[tid] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * P3M_SORT_TILE;
    uint32_t key[kItems];
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        const int64_t idx = base + r * kThreads + tid;
        key[r] = idx < n ? keys[idx] : 0u;
    }
#pragma unroll
    for (int r = 0; r < kItems; ++r)
        count_digit(hist, (key[r] >> shift) & (kRadix - 1), base + r * kThreads + tid < n, lane);
    __syncthreads();
    counts[(size_t)tid * n_tiles + blockIdx.x] = hist[tid];
}

__global__ void __launch_bounds__(kThreads)
    k_radix_downsweep(const uint32_t *__restrict__ keys_in, const uint32_t *__restrict__ vals_in,
                      int64_t n, int shift, const uint32_t *__restrict__ offsets, int n_tiles,
                      uint32_t *__restrict__ keys_out, uint32_t *__restrict__ vals_out)
{
    __shared__ uint32_t s_base[kRadix];
    __shared__ uint32_t s_cnt[kThreads / 32][kRadix];
    __shared__ uint32_t s_pos[kThreads / 32][kRadix];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    s_base[tid] = offsets[(size_t)tid * n_tiles + blockIdx.x];
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) s_cnt[w][tid] = 0;
    __syncthreads();
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t base = (int64_t)blockIdx.x * P3M_SORT_TILE;
    for (int r = 0; r < kItems; ++r) {
        const int64_t idx = base + r * kThreads + tid;
        const bool valid = idx < n;
        uint32_t key = 0, val = 0;
        if (valid) {
            key = keys_in[idx];
            val = vals_in ? vals_in[idx] : (uint32_t)idx;
        }
        const uint32_t d = (key >> shift) & (kRadix - 1);
        const uint32_t peers = match_digit(d, valid, kRadixBits);
        const uint32_t rank = __popc(peers & lt);
        if (valid && rank == 0) s_cnt[warp][d] = __popc(peers);
        __syncthreads();
        {
            uint32_t run = s_base[tid];
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) {
                const uint32_t c = s_cnt[w][tid];
                s_cnt[w][tid] = 0;
                s_pos[w][tid] = run;
                run += c;
            }
            s_base[tid] = run;
        }
        __syncthreads();
        if (valid) {
            const uint32_t p = s_pos[warp][d] + rank;
            keys_out[p] = key;
            vals_out[p] = val;
        }
    }
}

// ------------------------------------------------------------------ one-sweep LSD radix sort
// The particle sort of few keys: the digit counts of all passes from the keys' kernel, then one
// kernel per 8-bit pass.  A pass's CTAs take tiles (4096 keys, fewer for few particles) in launch
// order from an atomic counter; each ranks its tile (warp w its w-th eighth, round by round and lane
// by lane, so ranks are stable), publishes its per-digit counts, and finds the count of each digit in all earlier
// tiles by walking back over their published values (decoupled look-back: an entry holds a
// tile's own count, flag kAgg, or the running total through that tile, flag kInc).  A tile
// publishes kAgg before it waits for anything, and waits only on tiles taken before it, so
// every wait ends; each is still bounded (about a second) and sets P3M_FLAG_TIMEOUT when it
// gives up.  The tile is then reordered in shared memory by digit and written out in runs,
// coalesced, at global position = (keys of smaller digits) + (keys of the digit in earlier
// tiles) + (rank in the tile).
// Above P3M_SORT_SMALL keys a pass first counts every tile's digits and scans the counts instead: with
// hundreds of tiles in flight a tile looks back over hundreds of entries of 256 digits, and that traffic
// took more time than reading the keys twice.  Sort phase, before / now: 256^3 0.75 / 0.54 ms (look-back
// with eight entries at once: 0.63), 128^3 0.165 / 0.123, 48^3 (look-back, tiles of 1024; counting: 87 us)
// 50 / 35 us, 5003 keys 43 / 22 us (with the digit counts, which the keys' kernel has since taken over).  What bounds a pass now is the ranking: 26 ballots per key and their
// integer operations keep the ALU pipe 75 % busy.

constexpr int kWarps = kThreads / 32;
constexpr int kLookBack = 8;  // earlier tiles whose entries are read at once (a chain of single reads before)
constexpr uint32_t kAgg = 1u << 30, kInc = 2u << 30, kCountMask = kAgg - 1;  // (fewer than 2^30 keys)

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *total);

// kTileItems: keys per thread.  kChain: the counts of earlier tiles by look-back (hist: the digits' totals);
// otherwise hist holds, digit by digit, the first position of every tile's keys.
template <int kTileItems, bool kChain>
__global__ void __launch_bounds__(kThreads, 3)
    k_onesweep(const uint32_t *__restrict__ kin, const uint32_t *__restrict__ vin, int64_t n,
               int shift, int bits, const uint32_t *__restrict__ hist, uint32_t *status,
               uint32_t *tile_counter, uint32_t *__restrict__ kout, uint32_t *__restrict__ vout,
               uint32_t *flags, const uint32_t *lookback, long long wait_limit)
{
    constexpr int kTile = kTileItems * kThreads, kWarpItems = kTileItems * 32;
    __shared__ uint32_t s_key[kTile];
    __shared__ uint32_t s_val[kTile];
    __shared__ uint32_t s_wcnt[kWarps][kRadix];  // per-warp digit counts, then offsets
    __shared__ uint32_t s_off[kRadix];           // first tile slot of each digit
    __shared__ uint32_t s_out[kRadix];           // global position of the digit's first key
    __shared__ uint32_t s_tile;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_tile = kChain ? atomicAdd(tile_counter, 1u) : blockIdx.x;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) s_wcnt[w][tid] = 0;
    __syncthreads();
    const uint32_t tile = s_tile;
    if (tile >= gridDim.x) return;  // (never: the counter starts at zero)
    const int64_t wbase = (int64_t)tile * kTile + (int64_t)warp * kWarpItems;
    const uint32_t lt = (1u << lane) - 1u;

    // the warp's 512 keys and values (all loads in flight at once), then their ranks
    uint32_t key[kTileItems], val[kTileItems], rank[kTileItems];
#pragma unroll
    for (int r = 0; r < kTileItems; ++r) {
        const int64_t idx = wbase + r * 32 + lane;
        const bool valid = idx < n;
        key[r] = valid ? kin[idx] : 0u;
        val[r] = valid ? (vin ? vin[idx] : (uint32_t)idx) : 0u;
    }
#pragma unroll
    for (int r = 0; r < kTileItems; ++r) {
        const bool valid = wbase + r * 32 + lane < n;
        const uint32_t d = (key[r] >> shift) & (kRadix - 1);
        const uint32_t peers = match_digit(d, valid, bits);
        const int lead = __ffs(peers) - 1;
        uint32_t before = 0;
        if (valid && lane == lead) {
            before = s_wcnt[warp][d];
            s_wcnt[warp][d] = before + __popc(peers);
        }
        before = __shfl_sync(0xffffffffu, before, lead);
        rank[r] = before + __popc(peers & lt);
        __syncwarp();
    }
    __syncthreads();

    // thread tid = digit d: the tile's count, published at once; per-warp offsets
    const int d = tid;
    uint32_t cnt = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const uint32_t c = s_wcnt[w][d];
        s_wcnt[w][d] = cnt;
        cnt += c;
    }
    uint32_t *mine = status + (size_t)tile * kRadix + d;
    if (kChain) atomicExch(mine, (tile == 0 ? kInc : kAgg) | cnt);
    s_off[d] = block_exclusive_scan(cnt, nullptr);
    const uint32_t first = kChain ? block_exclusive_scan(hist[d], nullptr) : hist[(size_t)d * gridDim.x + tile];
    // keys of digit d in the tiles before this one
    uint32_t before = 0;
    if (kChain && tile > 0) {
        long long t = (long long)tile - 1;
        const long long t0 = clock64();
        for (bool done = false; !done;) {
            // lookback is status itself, except under an injected timeout (a zeroed copy)
            uint32_t v[kLookBack], any = 0, all = kAgg, sum = 0;
#pragma unroll
            for (int q = 0; q < kLookBack; ++q) {  // (before tile 0, which publishes kInc: never used)
                v[q] = t >= q ? *(const volatile uint32_t *)(lookback + (size_t)(t - q) * kRadix + d) : kInc;
                any |= v[q];
                all &= v[q];
                sum += v[q] & kCountMask;
            }
            int used = 0;
            if (!(any & kInc) && all) {  // all of them published, none with a running total
                before += sum;
                used = kLookBack;
            } else {
                bool ready = true;
#pragma unroll
                for (int q = 0; q < kLookBack; ++q) {
                    ready = ready && !done && (v[q] & ~kCountMask) != 0;
                    if (!ready) continue;
                    before += v[q] & kCountMask;
                    done = (v[q] & kInc) != 0;
                    ++used;
                }
            }
            t -= used;
            if (used == 0) {
                if (clock64() - t0 > wait_limit) {
                    atomicOr(flags, P3M_FLAG_TIMEOUT);
                    break;
                }
                __nanosleep(32);
            }
        }
        atomicExch(mine, kInc | (before + cnt));
    }
    s_out[d] = first + before;
    __syncthreads();

    // the tile in digit order in shared memory, then written out in runs
#pragma unroll
    for (int r = 0; r < kTileItems; ++r) {
        const int64_t idx = wbase + r * 32 + lane;
        if (idx < n) {
            const uint32_t dd = (key[r] >> shift) & (kRadix - 1);
            const uint32_t slot = s_off[dd] + s_wcnt[warp][dd] + rank[r];
            s_key[slot] = key[r];
            s_val[slot] = val[r];
        }
    }
    __syncthreads();
    const int64_t left = n - (int64_t)tile * kTile;
    const int count = left < kTile ? (int)left : kTile;
    for (int j = tid; j < count; j += kThreads) {
        const uint32_t k = s_key[j];
        const uint32_t dd = (k >> shift) & (kRadix - 1);
        const uint32_t p = s_out[dd] + (uint32_t)j - s_off[dd];
        if (p < n) {  // (always, unless a look-back wait gave up)
            kout[p] = k;
            vout[p] = s_val[j];
        }
    }
}

// ------------------------------------------------------------------ exclusive scan (uint32)

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *total)
{
    __shared__ uint32_t warp_sums[kThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t s = lane < kThreads / 32 ? warp_sums[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < kThreads / 32) warp_sums[lane] = s;
    }
    __syncthreads();
    const uint32_t before = warp ? warp_sums[warp - 1] : 0u;
    if (total) *total = warp_sums[kThreads / 32 - 1];
    __syncthreads();
    return before + x - v;
}

__global__ void __launch_bounds__(kThreads)
    k_scan_reduce(const uint32_t *__restrict__ in, size_t n, uint32_t *__restrict__ aux)
{
    const size_t base = (size_t)blockIdx.x * P3M_SORT_TILE;
    uint32_t s = 0;
    for (int r = 0; r < kItems; ++r) {
        const size_t i = base + r * kThreads + threadIdx.x;
        if (i < n) s += in[i];
    }
    uint32_t total;
    block_exclusive_scan(s, &total);
    if (threadIdx.x == 0) aux[blockIdx.x] = total;
}

// Single block: exclusive scan of aux[0..nb) in place, aux[nb] = total.
__global__ void __launch_bounds__(kThreads) k_scan_aux(uint32_t *aux, size_t nb)
{
    uint32_t carry = 0;
    for (size_t base = 0; base < nb; base += kThreads) {
        const size_t i = base + threadIdx.x;
        const uint32_t v = i < nb ? aux[i] : 0u;
        uint32_t total;
        const uint32_t ex = block_exclusive_scan(v, &total);
        if (i < nb) aux[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) aux[nb] = carry;
}

// Each thread owns 16 consecutive items of the block's 4096 (read before any write, so
// in == out is allowed).
__global__ void __launch_bounds__(kThreads)
    k_scan_down(const uint32_t *in, uint32_t *out, size_t n, const uint32_t *__restrict__ aux)
{
    const size_t base = (size_t)blockIdx.x * P3M_SORT_TILE + (size_t)threadIdx.x * kItems;
    uint32_t v[kItems];
    uint32_t s = 0;
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        v[r] = (base + r < n) ? in[base + r] : 0u;
        s += v[r];
    }
    uint32_t run = aux[blockIdx.x] + block_exclusive_scan(s, nullptr);
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        if (base + r < n) out[base + r] = run;
        run += v[r];
    }
}

// ------------------------------------------------------------------ permutation and cells

template <typename R4>
__device__ __forceinline__ R4 make_rel(double x, double y, double z);
template <>
__device__ __forceinline__ float4 make_rel<float4>(double x, double y, double z)
{
    return make_float4((float)x, (float)y, (float)z, 0.0f);
}
template <>
__device__ __forceinline__ double4_16a make_rel<double4_16a>(double x, double y, double z)
{
    return make_double4_16a(x, y, z, 0.0);
}

// FP32 mode: position minus its cell origin (no FP32 absolute coordinate).  FP64 mode: the
// absolute position itself, so that the pair kernel forms x_j - x_i exactly like a plain
// minimum-image difference.
// (origin[c] = c * cs, a host table: the same correctly rounded products without the FP64
// multiply and conversion per particle)
template <typename R4>
__device__ __forceinline__ R4 rel_coords(double x, double y, double z, uint32_t cx, uint32_t cy,
                                         uint32_t cz, const double *origin)
{
    return make_rel<R4>(x - __ldg(origin + cx), y - __ldg(origin + cy), z - __ldg(origin + cz));
}
template <>
__device__ __forceinline__ double4_16a rel_coords<double4_16a>(double x, double y, double z, uint32_t,
                                                       uint32_t, uint32_t, const double *)
{
    return make_double4_16a(x, y, z, 0.0);
}

// One warp per 32-slot block of the sorted order; with kPairs (a context with the short-range force)
// the warp also writes the block's fixed-point coordinates and its bounding box (FP32, absolute
// coordinates, within the margins of the culling radii).
// What bounds it: reads of particles in the caller's order, 8 bytes at a time (3 GB of DRAM reads at
// 256^3 where 1 GB is asked for, 80 % of the DRAM throughput), and 9 FP64 operations per particle (6
// without kPairs, before 12).  Six CTAs per SM (40 registers): 0.644 -> 0.619 ms at 256^3 against five.
// Pure PM, 256^3: 0.727 -> 0.678 ms.
template <typename R4, bool kPairs>
__global__ void __launch_bounds__(256, 6) k_permute(const uint32_t *__restrict__ perm, const uint32_t *__restrict__ keys,
                          P3MGeom g, const double *__restrict__ pos,
                          const double *__restrict__ mom, const uint32_t *__restrict__ pid,
                          double *__restrict__ pos_out, double *__restrict__ mom_out,
                          uint32_t *__restrict__ pid_out, R4 *__restrict__ rel,
                          float4 *__restrict__ block_box, uint32_t *__restrict__ relq, double fix_scale,
                          const double *__restrict__ origin, uint32_t *__restrict__ cell_start)
{
    constexpr bool kFp32 = sizeof(R4) == sizeof(float4);
    const float cs = (float)g.cs;
    const int64_t n = g.n;
    const int64_t nblocks = (n + 31) >> 5;
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t blk = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; blk < nblocks;
         blk += nwarps) {
        const int64_t k = blk * 32 + lane;
        const bool active = k < n;
        const uint32_t pj = perm[active ? k : blk * 32];
        p3m_in_bounds(pj < (uint32_t)n, g.flags);
        const uint32_t j = min(pj, (uint32_t)(n - 1));  // in bounds always
        const double x = pos[j], y = pos[n + j], z = pos[2 * n + j];
        R4 rv = make_rel<R4>(0.0, 0.0, 0.0);
        float lx = 0.0f, ly = 0.0f, lz = 0.0f;
        if (active) {
            pos_out[k] = x;
            pos_out[n + k] = y;
            pos_out[2 * n + k] = z;
            mom_out[k] = mom[j];
            mom_out[n + k] = mom[n + j];
            mom_out[2 * n + k] = mom[2 * n + j];
            pid_out[k] = pid[j];
            const uint32_t cell = cell_of_key(keys[k], g.sub_bits, g.n_cells);
            p3m_in_bounds((keys[k] >> (3 * g.sub_bits)) < (uint32_t)g.n_cells, g.flags);
            first_slots(keys, k, cell, n, g.sub_bits, g.n_cells, cell_start);
            const uint32_t cx = cell % g.n_c, cy = (cell / g.n_c) % g.n_c,
                           cz = cell / (g.n_c * g.n_c);
            rv = rel_coords<R4>(x, y, z, cx, cy, cz, origin);
            if (kFp32 || kPairs) rel[k] = rv;
            if (kFp32) {
                lx = fmaf((float)cx, cs, (float)rv.x);
                ly = fmaf((float)cy, cs, (float)rv.y);
                lz = fmaf((float)cz, cs, (float)rv.z);
            }
        }
        if (!kPairs) continue;
        {  // fixed point: 1.5 * 2^52 rounds x * scale to an integer in the low word (modulo 2^32)
            uint32_t *fix = relq + blk * 96;
            fix[lane] = (uint32_t)__double_as_longlong(fma(x, fix_scale, 0x1.8p52));
            fix[32 + lane] = (uint32_t)__double_as_longlong(fma(y, fix_scale, 0x1.8p52));
            fix[64 + lane] = (uint32_t)__double_as_longlong(fma(z, fix_scale, 0x1.8p52));
        }
        if (!kFp32) {
            lx = (float)x;
            ly = (float)y;
            lz = (float)z;
        }
        // (slots past the end stand for the block's first particle)
        const float l0 = __shfl_sync(0xffffffffu, lx, 0), l1 = __shfl_sync(0xffffffffu, ly, 0),
                    l2 = __shfl_sync(0xffffffffu, lz, 0);
        if (!active) lx = l0, ly = l1, lz = l2;
        float hx = lx, hy = ly, hz = lz;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lx = fminf(lx, __shfl_xor_sync(0xffffffffu, lx, o));
            ly = fminf(ly, __shfl_xor_sync(0xffffffffu, ly, o));
            lz = fminf(lz, __shfl_xor_sync(0xffffffffu, lz, o));
            hx = fmaxf(hx, __shfl_xor_sync(0xffffffffu, hx, o));
            hy = fmaxf(hy, __shfl_xor_sync(0xffffffffu, hy, o));
            hz = fmaxf(hz, __shfl_xor_sync(0xffffffffu, hz, o));
        }
        if (lane == 0) {
            block_box[2 * blk] = make_float4(lx, ly, lz, 0.0f);
            block_box[2 * blk + 1] = make_float4(hx, hy, hz, 0.0f);
        }
    }
}

__global__ void k_cell_start(const uint32_t *__restrict__ keys, P3MGeom g,
                             uint32_t *__restrict__ cell_start)
{
    const int64_t n = g.n;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x)
        first_slots(keys, k, cell_of_key(keys[k], g.sub_bits, g.n_cells), n, g.sub_bits, g.n_cells, cell_start);
}

// The pair work list (work_list.h): items of up to 32 particles of one cell, work[2w] = cell, work[2w + 1] =
// first slot, the most expensive first.  An item's cost estimate is (its particles) x (particles in the 27 neighbour
// cells); its key is the class log2(cost) to 1/8 octave (the FP32 exponent and top 3 mantissa bits, 8 bits),
// inverted.  k_work_count counts the items of every class, k_work_place scans the 256 counts and gives each
// item a place in its class (their order within a class is arbitrary: results do not depend on it).  Two
// kernels instead of a count, a scan, a fill and a radix pass with its memsets (ten launches and memsets):
// 5003 particles 23 -> 8 us of kernels, clustered 128^3 (a thread wrote all items of a dense cell; now its
// warp does) 55 -> 12 us.

// hist[key] += items (pairs), *max_count = max particles of a cell
__global__ void __launch_bounds__(kThreads)
    k_work_count(const uint32_t *__restrict__ cell_start, int n_c, int n_cells, bool pairs,
                 uint32_t *__restrict__ hist, uint32_t *__restrict__ max_count)
{
    __shared__ uint32_t h[kRadix];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int c = blockIdx.x * kThreads + threadIdx.x;
    uint32_t count = 0;
    if (c < n_cells) {
        const uint32_t s0 = cell_start[c], s1 = cell_start[c + 1];
        count = s1 > s0 ? s1 - s0 : 0u;
        if (pairs && count) {
            const WorkItems w = work_items(cell_start, n_c, c);
            if (w.full) atomicAdd(&h[w.key_full], w.full);
            if (w.rest) atomicAdd(&h[w.key_rest], 1u);
        }
    }
    const uint32_t most = __reduce_max_sync(0xffffffffu, count);
    if ((threadIdx.x & 31) == 0 && most) atomicMax(max_count, most);
    __syncthreads();
    if (h[threadIdx.x]) atomicAdd(hist + threadIdx.x, h[threadIdx.x]);
}

// hist: the classes' items; next (zeroed): places taken so far.  work_key: the keys, 0xFFFFFFFF after the
// last item (ensembles sort several contexts' lists together).
__global__ void __launch_bounds__(kThreads)
    k_work_place(const uint32_t *__restrict__ cell_start, int n_c, int n_cells, const uint32_t *__restrict__ hist,
                 uint32_t *__restrict__ next, uint32_t *__restrict__ n_work, size_t max_work,
                 uint2 *__restrict__ work, uint32_t *__restrict__ work_key)
{
    __shared__ uint32_t mine[kRadix], base[kRadix];
    const int tid = threadIdx.x, lane = tid & 31;
    mine[tid] = 0;
    __syncthreads();
    const int c = blockIdx.x * kThreads + tid;
    WorkItems w = {0u, 0u, 0u, 255u, 255u};
    if (c < n_cells) w = work_items(cell_start, n_c, c);
    uint32_t at_full = w.full ? atomicAdd(&mine[w.key_full], w.full) : 0u;
    uint32_t at_rest = w.rest ? atomicAdd(&mine[w.key_rest], 1u) : 0u;
    __syncthreads();
    uint32_t total;
    const uint32_t before = block_exclusive_scan(hist[tid], &total);
    base[tid] = before + (mine[tid] ? atomicAdd(next + tid, mine[tid]) : 0u);
    total = work_length(total, max_work);
    if (blockIdx.x == 0 && tid == 0) *n_work = total;
    __syncthreads();
    at_full += base[w.key_full];
    at_rest += base[w.key_rest];
    auto put = [&](uint32_t at, int cell, uint32_t slot, uint32_t key) {
        if (at >= max_work) return;  // (never, unless a sort gave up)
        work[at] = make_uint2((uint32_t)cell, slot);
        work_key[at] = key;
    };
    constexpr uint32_t kOwn = 16;  // a lane's own cell up to this many items, more by the whole warp
    if (w.full <= kOwn)
        for (uint32_t i = 0; i < w.full; ++i) put(at_full + i, c, w.first + i * P3M_PAIR_TI, w.key_full);
    if (w.rest) put(at_rest, c, w.first + w.full * P3M_PAIR_TI, w.key_rest);
    for (uint32_t m = __ballot_sync(0xffffffffu, w.full > kOwn); m; m &= m - 1) {
        const int l = __ffs(m) - 1;
        const uint32_t full = __shfl_sync(0xffffffffu, w.full, l), at = __shfl_sync(0xffffffffu, at_full, l);
        const uint32_t first = __shfl_sync(0xffffffffu, w.first, l), key = __shfl_sync(0xffffffffu, w.key_full, l);
        const int cell = __shfl_sync(0xffffffffu, c, l);
        for (uint32_t i = lane; i < full; i += 32) put(at + i, cell, first + i * P3M_PAIR_TI, key);
    }
    for (size_t i = total + blockIdx.x * (size_t)kThreads + tid; i < max_work; i += (size_t)gridDim.x * kThreads)
        work_key[i] = 0xFFFFFFFFu;
}

inline int grid_for(int64_t n, int threads, int num_sms)
{
    int64_t b = (n + threads - 1) / threads;
    int64_t cap = (int64_t)num_sms * 16;
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

namespace {

// How the particle sort of a context runs: by look-back (few particles; an injected timeout needs a look-back
// to wait in) or counted passes.  The keys' kernel clears and fills the look-back's digit counts, so
// every look-back sort follows one.
struct SortPlan {
    bool small, chain;
    int passes;
    unsigned n_tiles;
    size_t status_words;  // look-back entries of a pass
};

SortPlan sort_plan(const p3m_ctx *c)
{
    SortPlan p;
    p.small = c->g.n <= P3M_SORT_SMALL;
    p.chain = p.small || c->sort_probe;
    p.passes = (c->key_bits + kRadixBits - 1) / kRadixBits;
    const int64_t tile = p.small ? 4 * kThreads : P3M_SORT_TILE;
    p.n_tiles = (unsigned)((c->g.n + tile - 1) / tile);
    p.status_words = (size_t)kRadix * p.n_tiles;
    return p;
}

}  // namespace

cudaError_t launch_kick_drift_keys(p3m_ctx *c, bool kick_drift, double kfac, double dfac,
                                   bool from_table)
{
    const SortPlan sp = sort_plan(c);
    if (sp.chain) {
        // sort_hist: 4 x 256 digit counts, then one tile counter per pass; sort_status follows it.  Few
        // particles have a status array per pass, cleared together.
        const cudaError_t e = cudaMemsetAsync(
            c->sort_hist, 0, P3M_SORT_HIST_BYTES + 4 * sp.status_words * (sp.small ? sp.passes : 1), c->stream);
        if (e != cudaSuccess) return e;
    }
    c->launches += 1;
    auto pick = [&](auto bits) {
        constexpr int kB = decltype(bits)::value;
        return kick_drift ? (sp.chain ? k_kick_drift_keys<kB, true, true> : k_kick_drift_keys<kB, true, false>)
                          : (sp.chain ? k_kick_drift_keys<kB, false, true> : k_kick_drift_keys<kB, false, false>);
    };
    auto kern = c->g.sub_bits == 3 ? pick(std::integral_constant<int, 3>{}) : pick(std::integral_constant<int, -1>{});
    kern<<<grid_for(c->g.n, kThreads, c->num_sms), kThreads, 0, c->stream>>>(
        c->pos, c->mom, c->acc, c->g, kfac, dfac, c->keys, from_table ? c->cur_fac : nullptr, sp.passes, c->sort_hist);
    return cudaGetLastError();
}

cudaError_t launch_scan_u32(const uint32_t *in, uint32_t *out, size_t n, uint32_t *aux,
                            cudaStream_t s)
{
    const size_t nb = (n + P3M_SORT_TILE - 1) / P3M_SORT_TILE;
    if (nb == 0) return cudaSuccess;
    k_scan_reduce<<<(unsigned)nb, kThreads, 0, s>>>(in, n, aux);
    k_scan_aux<<<1, kThreads, 0, s>>>(aux, nb);
    k_scan_down<<<(unsigned)nb, kThreads, 0, s>>>(in, out, n, aux);
    return cudaGetLastError();
}

// Stable LSD sort of n (key, value) pairs on the low key_bits bits.  k[0]/v[0] hold the input
// (v[0] NULL: values are the input positions); on return k[0]/v[0] hold the sorted pairs (the
// two buffers of each array are swapped as needed).  counts needs 256 * ceil(n/4096) entries.
cudaError_t radix_sort_pairs(uint32_t **k, uint32_t **v, bool identity_vals, int64_t n,
                             int key_bits, uint32_t *counts, uint32_t *aux, cudaStream_t s,
                             unsigned long long *launches)
{
    const int passes = (key_bits + kRadixBits - 1) / kRadixBits;
    const int n_tiles = (int)((n + P3M_SORT_TILE - 1) / P3M_SORT_TILE);
    const size_t ncount = (size_t)kRadix * n_tiles;
    uint32_t *kin = k[0], *kout = k[1];
    uint32_t *vin = identity_vals ? nullptr : v[0], *vout = identity_vals ? v[0] : v[1];
    for (int p = 0; p < passes; ++p) {
        const int shift = p * kRadixBits;
        *launches += 5;  // upsweep, 3 scan kernels, downsweep
        k_radix_upsweep<<<n_tiles, kThreads, 0, s>>>(kin, n, shift, counts, n_tiles);
        cudaError_t e = launch_scan_u32(counts, counts, ncount, aux, s);
        if (e != cudaSuccess) return e;
        k_radix_downsweep<<<n_tiles, kThreads, 0, s>>>(kin, vin, n, shift, counts, n_tiles, kout,
                                                       vout);
        uint32_t *t = kin;  // the next pass reads what this one wrote
        kin = kout;
        kout = t;
        uint32_t *vt = vin;
        vin = vout;
        vout = vt ? vt : v[1];
    }
    if (kin != k[0]) {
        k[1] = k[0];
        k[0] = kin;
    }
    if (vin != v[0]) {
        v[1] = v[0];
        v[0] = vin;
    }
    return cudaGetLastError();
}

cudaError_t launch_radix_sort(p3m_ctx *c)
{
    const int64_t n = c->g.n;
    const SortPlan sp = sort_plan(c);
    const bool small = sp.small, chain = sp.chain;
    const int passes = sp.passes;
    const unsigned n_tiles = sp.n_tiles;
    const size_t status_words = sp.status_words;
    cudaStream_t s = c->stream;
    cudaError_t e = cudaSuccess;
    for (int p = 0; p < passes; ++p) {
        const int shift = p * kRadixBits, bits = min(kRadixBits, c->key_bits - shift);
        const uint32_t *vin = p ? c->vals : nullptr;  // the first pass's values are the slots
        if (chain) {
            uint32_t *status = c->sort_status + (small ? p * status_words : 0);
            if (!small && p > 0) e = cudaMemsetAsync(status, 0, 4 * status_words, s);
            if (e != cudaSuccess) return e;
            auto sweep = small ? k_onesweep<4, true> : k_onesweep<kItems, true>;
            sweep<<<n_tiles, kThreads, 0, s>>>(c->keys, vin, n, shift, bits, c->sort_hist + p * kRadix, status,
                                               c->sort_hist + 4 * kRadix + p, c->keys_alt, c->vals_alt,
                                               c->counters + 1, c->sort_probe ? c->sort_probe : status,
                                               c->sort_wait_limit);
        } else {
            k_radix_upsweep<<<n_tiles, kThreads, 0, s>>>(c->keys, n, shift, c->digit_counts, n_tiles);
            e = launch_scan_u32(c->digit_counts, c->digit_counts, status_words, c->scan_aux, s);
            if (e != cudaSuccess) return e;
            k_onesweep<kItems, false><<<n_tiles, kThreads, 0, s>>>(c->keys, vin, n, shift, bits, c->digit_counts,
                                                                   nullptr, nullptr, c->keys_alt, c->vals_alt,
                                                                   nullptr, nullptr, 0);
            c->launches += 4;
        }
        c->launches += 1;
        uint32_t *t = c->keys;  // the next pass reads what this one wrote
        c->keys = c->keys_alt;
        c->keys_alt = t;
        t = c->vals;
        c->vals = c->vals_alt;
        c->vals_alt = t;
    }
    return cudaGetLastError();
}

cudaError_t launch_permute_and_cells(p3m_ctx *c)
{
    const int64_t n = c->g.n;
    const int gb = grid_for(n, 256, c->num_sms);
    const double fix_scale = ldexp((double)c->g.n_c, kFixBits) / c->g.box;
    c->launches += 2;  // permute, work_count
    auto permute = [&](auto kern, auto *rel) {
        kern<<<gb, 256, 0, c->stream>>>(c->vals, c->keys, c->g, c->pos, c->mom, c->pid, c->pos_alt, c->mom_alt,
                                        c->pid_alt, rel, c->block_box, c->relq, fix_scale, c->tab_origin, c->cell_start);
    };
    if (c->precision == P3M_PREC_MIXED)
        permute(c->short_range ? k_permute<float4, true> : k_permute<float4, false>, (float4 *)c->rel);
    else
        permute(c->short_range ? k_permute<double4_16a, true> : k_permute<double4_16a, false>, (double4_16a *)c->rel);
    double *t = c->pos;
    c->pos = c->pos_alt;
    c->pos_alt = t;
    t = c->mom;
    c->mom = c->mom_alt;
    c->mom_alt = t;
    uint32_t *u = c->pid;
    c->pid = c->pid_alt;
    c->pid_alt = u;

    // counters: [2] max cell count, [3] spare, [4 ..] 256 class counts, the number of items, 256 places
    cudaError_t e = cudaMemsetAsync(c->counters + 2, 0, sizeof(uint32_t) * (P3M_COUNTERS - 2), c->stream);
    if (e != cudaSuccess) return e;
    const unsigned gc = (unsigned)((c->g.n_cells + kThreads - 1) / kThreads);
    uint32_t *hist = c->counters + 4, *next = c->n_work + 1;
    k_work_count<<<gc, kThreads, 0, c->stream>>>(c->cell_start, c->g.n_c, c->g.n_cells, c->short_range != 0, hist,
                                                 c->counters + 2);
    if (c->short_range) {
        c->launches += 1;
        k_work_place<<<gc, kThreads, 0, c->stream>>>(c->cell_start, c->g.n_c, c->g.n_cells, hist, next, c->n_work,
                                                     c->max_work, (uint2 *)c->work, c->work_key);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------ allocation-free binning
// p3m_cell_sort_noalloc: the chaining-cell keys, stable sort and cell ranges of the context's
// force evaluation, for callers that must not allocate device memory.  Its scratch (two key
// arrays, the spare value array, the radix digit counts and the scan partials) is one
// file-scope device array, sized for at most P3M_NOALLOC_MAX_N particles; every GPU that loads
// the library holds it until the process exits.

namespace {

constexpr int64_t kNoAllocMaxN = P3M_NOALLOC_MAX_N;
constexpr int kNoAllocTiles = (int)((kNoAllocMaxN + P3M_SORT_TILE - 1) / P3M_SORT_TILE);
constexpr size_t kNoAllocCounts = (size_t)kRadix * kNoAllocTiles;
constexpr size_t kNoAllocAux = kNoAllocCounts / P3M_SORT_TILE + 8;
constexpr size_t kNoAllocWords = 3 * (size_t)kNoAllocMaxN + kNoAllocCounts + kNoAllocAux;

// Keys of positions that stay unmodified: the same wrap and key arithmetic as
// k_kick_drift_keys, without writing the positions back.
__global__ void k_keys_only(const double *__restrict__ pos, P3MGeom g, uint32_t *__restrict__ keys)
{
    const int64_t n = g.n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t f[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) f[d] = fine_index(wrap_box(pos[d * n + i], g.box), g.inv_fine, g.n_fine);
        keys[i] = make_key<-1>(f[0], f[1], f[2], g);
    }
}

}  // namespace

static __device__ __align__(256) uint32_t g_noalloc_scratch[kNoAllocWords];

namespace {

std::mutex g_noalloc_mutex;
uint32_t *g_noalloc_ptr[256];  // device address of g_noalloc_scratch, per device ordinal

// Device address of the scratch on the current device, looked up with that device current (the
// host-side symbol itself is not a device address).  The first call on a device must look it up
// outside stream capture; later calls look it up again whenever the stream is not capturing, so
// that an address cached before a cudaDeviceReset (which reloads the module in a new context) is
// never used afterwards; while capturing they use the cached address.
cudaError_t noalloc_scratch(cudaStream_t stream, uint32_t **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(stream, &cap);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (cap == cudaStreamCaptureStatusNone) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = (uint32_t *)p;
    } else if (!g_noalloc_ptr[dev]) {
        return cudaErrorStreamCaptureUnsupported;  // no set-up call before the capture began
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}

}  // namespace

extern "C" int p3m_cell_sort_noalloc(const double *pos3n, int64_t n, double box, int n_c,
                                     int sub_bits, uint32_t *keys_out, uint32_t *ids_out,
                                     uint32_t *cell_start_out, void *stream)
{
    if (!pos3n || !keys_out || !ids_out || !cell_start_out)
        return p3m_fail_global(P3M_EINVAL, "p3m_cell_sort_noalloc: NULL pointer argument");
    if (n < 1 || n > kNoAllocMaxN)
        return p3m_fail_global(P3M_EINVAL,
                               "p3m_cell_sort_noalloc: n = %lld outside [1, %lld] (fixed scratch size)",
                               (long long)n, (long long)kNoAllocMaxN);
    if (!(box > 0.0) || !isfinite(box) || n_c < 1 || n_c > 1024 || sub_bits < 0 || sub_bits > 3)
        return p3m_fail_global(P3M_EINVAL, "p3m_cell_sort_noalloc: need box > 0, 1 <= n_c <= 1024, "
                                           "0 <= sub_bits <= 3");
    const uint64_t max_key = ((uint64_t)n_c * n_c * n_c << (3 * sub_bits)) - 1;
    if (max_key >= (1ull << 32))
        return p3m_fail_global(P3M_EINVAL, "p3m_cell_sort_noalloc: sort key exceeds 32 bits");
    int key_bits = 1;
    while (key_bits < 32 && (max_key >> key_bits)) ++key_bits;

    uint32_t *scratch = nullptr;
    cudaError_t e = noalloc_scratch((cudaStream_t)stream, &scratch);
    if (e != cudaSuccess)
        return p3m_fail_global(P3M_ECUDA, "p3m_cell_sort_noalloc: scratch lookup failed: %s",
                               cudaGetErrorString(e));
    uint32_t *keys0 = scratch, *keys1 = scratch + kNoAllocMaxN, *vals1 = scratch + 2 * kNoAllocMaxN;
    uint32_t *counts = scratch + 3 * kNoAllocMaxN, *aux = counts + kNoAllocCounts;

    P3MGeom g;
    memset(&g, 0, sizeof(g));
    g.box = box;
    g.n = n;
    g.n_c = n_c;
    g.sub_bits = sub_bits;
    g.n_fine = n_c << sub_bits;
    g.inv_fine = (double)g.n_fine / box;
    g.n_cells = n_c * n_c * n_c;
    cudaStream_t s = (cudaStream_t)stream;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);

    k_keys_only<<<grid_for(n, 256, sms), 256, 0, s>>>(pos3n, g, keys0);
    unsigned long long launches = 0;
    uint32_t *k[2] = {keys0, keys1}, *v[2] = {ids_out, vals1};
    e = radix_sort_pairs(k, v, true, n, key_bits, counts, aux, s, &launches);
    if (e == cudaSuccess) e = cudaMemcpyAsync(keys_out, k[0], 4 * (size_t)n, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess && v[0] != ids_out)
        e = cudaMemcpyAsync(ids_out, v[0], 4 * (size_t)n, cudaMemcpyDeviceToDevice, s);
    if (e == cudaSuccess) {
        k_cell_start<<<grid_for(n, 256, sms), 256, 0, s>>>(keys_out, g, cell_start_out);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess)
        return p3m_fail_global(P3M_ECUDA, "p3m_cell_sort_noalloc: %s", cudaGetErrorString(e));
    return P3M_OK;
}
