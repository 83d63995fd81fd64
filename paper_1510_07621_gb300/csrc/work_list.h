// Cell ranges and pair work items from sorted keys, one particle or cell at a time: the parts of the
// kernels in sort.cu that must stay within their arrays whatever order the keys have.  A sort whose
// look-back gave up leaves any order (and keys of other sub_bits); the flag it sets is read by the host only
// at its next synchronisation, after the evaluation.  Compiles as plain C++ too, for tests without a GPU.
#pragma once

#include <stddef.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define P3M_HD __host__ __device__ __forceinline__
#else
#define P3M_HD static inline
#endif

constexpr uint32_t kWorkItem = 32;  // particles per work item

P3M_HD uint32_t cell_of_key(uint32_t key, int sub_bits, int n_cells)
{
    const uint32_t c = key >> (3 * sub_bits);
    return c < (uint32_t)n_cells ? c : (uint32_t)n_cells - 1u;
}

// cell_start[c] = first sorted slot whose cell is >= c, the part that slot k (of cell `cell`) writes:
// the cells after the previous slot's up to its own, and the last slot also the cells after its own.  Whatever
// the order, every entry is written by some slot, with a value in [0, n].
P3M_HD void first_slots(const uint32_t *keys, int64_t k, uint32_t cell, int64_t n, int sub_bits, int n_cells,
                        uint32_t *cell_start)
{
    const int64_t prev = k > 0 ? (int64_t)cell_of_key(keys[k - 1], sub_bits, n_cells) : -1;
    for (int64_t c = prev + 1; c <= (int64_t)cell; ++c) cell_start[c] = (uint32_t)k;
    if (k == n - 1)
        for (int64_t c = (int64_t)cell + 1; c <= (int64_t)n_cells; ++c) cell_start[c] = (uint32_t)n;
}

struct WorkItems {
    uint32_t first, full, rest;  // first slot, items of 32, particles of the last item
    uint32_t key_full, key_rest;
};

// An item's key: its cost's class, log2((particles) x (particles near)) to 1/8 octave, inverted
P3M_HD uint32_t work_key_of(uint32_t particles, uint32_t near)
{
    const float cost = (float)particles * (float)near;  // >= 1
    uint32_t bits;
    memcpy(&bits, &cost, sizeof(bits));
    const uint32_t cls = (bits >> 20) - (127u << 3);
    return 255u - (cls < 255u ? cls : 255u);
}

// the items of cell c (none where the ranges are not ordered)
P3M_HD WorkItems work_items(const uint32_t *cell_start, int n_c, int c)
{
    WorkItems w = {cell_start[c], 0u, 0u, 255u, 255u};
    const uint32_t end = cell_start[c + 1];
    if (end <= w.first) return w;
    const int cx = c % n_c, cy = (c / n_c) % n_c, cz = c / (n_c * n_c);
    // rows of three cells along x are consecutive slots (a row that wraps: the rest of it)
    uint32_t near = 0;
#ifdef __CUDACC__
#pragma unroll
#endif
    for (int oz = -1; oz <= 1; ++oz) {
        int z = cz + oz;
        z += z < 0 ? n_c : (z >= n_c ? -n_c : 0);
#ifdef __CUDACC__
#pragma unroll
#endif
        for (int oy = -1; oy <= 1; ++oy) {
            int y = cy + oy;
            y += y < 0 ? n_c : (y >= n_c ? -n_c : 0);
            const uint32_t *row = cell_start + ((size_t)z * n_c + y) * n_c;
            near += row[cx + 2 < n_c ? cx + 2 : n_c] - row[cx > 0 ? cx - 1 : 0];
            if (cx == 0) near += row[n_c] - row[n_c - 1];
            if (cx == n_c - 1) near += row[1] - row[0];
        }
    }
    w.full = (end - w.first) / kWorkItem;
    w.rest = (end - w.first) % kWorkItem;
    w.key_full = work_key_of(kWorkItem, near);
    if (w.rest) w.key_rest = work_key_of(w.rest, near);
    return w;
}

// The length of the list that the pair kernels read: ordered ranges never have more than max_work items,
// unordered ones may (their positive lengths add up to more than n); those at or beyond it are not stored.
P3M_HD uint32_t work_length(uint32_t items, size_t max_work)
{
    return items < max_work ? items : (uint32_t)max_work;
}
