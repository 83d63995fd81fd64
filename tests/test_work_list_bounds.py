"""The work list from keys in any order (csrc/work_list.h, compiled here as plain C++; CPU only): a sort whose
look-back gave up leaves the keys unordered, and the evaluation that follows must stay within its arrays.
Every cell_start entry is written, at most max_work items are listed, each entry up to the list's length is
written and names a cell and a slot that exist; an ordered set's list is complete."""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1510_07621_gb300", "csrc")

HARNESS = r"""
#include "work_list.h"
// the kernels of sort.cu, one particle (in any order: the writers race) and one cell after another
extern "C" uint32_t make_list(const uint32_t *keys, const int64_t *when, int64_t n, int sub_bits, int n_c, uint32_t *cell_start,
                              size_t max_work, uint32_t *work, uint32_t *items)
{
    const int n_cells = n_c * n_c * n_c;
    for (int64_t t = 0; t < n; ++t) {
        const int64_t k = when[t];
        first_slots(keys, k, cell_of_key(keys[k], sub_bits, n_cells), n, sub_bits, n_cells, cell_start);
    }
    uint32_t hist[256] = {0}, next[256], total = 0;
    for (int c = 0; c < n_cells; ++c) {
        const WorkItems w = work_items(cell_start, n_c, c);
        hist[w.key_full] += w.full;
        if (w.rest) hist[w.key_rest] += 1;
    }
    for (int q = 0; q < 256; ++q) {
        next[q] = total;
        total += hist[q];
    }
    *items = total;
    for (int c = 0; c < n_cells; ++c) {
        const WorkItems w = work_items(cell_start, n_c, c);
        auto put = [&](uint32_t at, uint32_t slot) {
            if (at >= max_work) return;
            work[2 * at] = (uint32_t)c;
            work[2 * at + 1] = slot;
        };
        for (uint32_t i = 0; i < w.full; ++i) put(next[w.key_full]++, w.first + i * kWorkItem);
        if (w.rest) put(next[w.key_rest]++, w.first + w.full * kWorkItem);
    }
    return work_length(total, max_work);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("work_list")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-std=c++17", "-I" + CSRC, str(d / "h.cpp"), "-o",
                    str(d / "h.so")], check=True)
    so = ctypes.CDLL(str(d / "h.so"))
    so.make_list.restype = ctypes.c_uint32
    return so


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("n,n_c", [(1, 3), (33, 3), (1000, 3), (4000, 5), (20000, 11)])
@pytest.mark.parametrize("order", ["sorted", "random", "two runs", "other sub_bits", "sawtooth"])
def test_list_stays_within_its_arrays(lib, n, n_c, order):
    rng = np.random.default_rng(n)
    sub_bits, cells = 2, n_c ** 3
    keys = np.sort(rng.integers(0, cells << (3 * sub_bits), n, dtype=np.uint32))
    if order == "random":
        keys = rng.permutation(keys)
    elif order == "two runs":
        keys = np.concatenate([keys[::2], keys[1::2]])
    elif order == "other sub_bits":
        keys = rng.permutation(keys << np.uint32(3))
    elif order == "sawtooth" and n > 4 * cells:  # every other cell seems to hold almost all particles
        up = np.arange(cells)
        pairs = np.stack([up[1::2] - 1, up[1::2]], axis=1)[::-1].reshape(-1)
        keys = np.concatenate([up, np.full(n - cells - pairs.size - 1, cells - 1), pairs, [cells - 1]])
        keys = (keys << (3 * sub_bits)).astype(np.uint32)
    when = rng.permutation(n) if order in ("random", "two runs", "other sub_bits") else np.arange(n)
    if order == "sawtooth":
        when = np.concatenate([[n - 1], np.arange(n - 1)])
    when = when.astype(np.int64)
    max_work = n // 32 + cells + 1
    start = np.full(cells + 1, 0xDEADBEEF, np.uint32)
    work = np.full(2 * max_work, 0xDEADBEEF, np.uint32)
    items = ctypes.c_uint32()
    count = lib.make_list(_ptr(keys), _ptr(when), ctypes.c_int64(n), sub_bits, n_c, _ptr(start), ctypes.c_size_t(max_work),
                          _ptr(work), ctypes.byref(items))
    assert np.all(start <= n) and start[-1] == n
    assert count <= max_work and count == min(items.value, max_work)
    cell, slot = work.reshape(-1, 2)[:count].astype(np.int64).T
    assert np.all(cell < cells) and np.all(slot < n)
    if order == "sorted":
        size = np.diff(start.astype(np.int64))
        assert size.sum() == n and count == int(((size + 31) // 32).sum())
    if order == "sawtooth" and n > 4 * cells:
        assert items.value > max_work  # the length has to be cut off
