"""The bit-level floor of a mesh coordinate (split_floor in csrc/state.cuh), emulated in numpy: integer part
and fraction equal floor(u) and u - floor(u) exactly for 0 <= u < 4096."""

import numpy as np
import pytest


def split_floor(u):
    b = u.view(np.uint64)
    e = (b >> np.uint64(52)).astype(np.int64) - 1023
    s = (e & 15).astype(np.uint64)
    frac = (b << s) & np.uint64(0xFFFFFFFFFFFFF)
    g = (frac | np.uint64(0x3FF0000000000000)).view(np.float64) - 1.0
    top = ((b >> np.uint64(32)) & np.uint64(0xFFFFF)) | np.uint64(0x100000)
    whole = (e >= 0) & (e < 12)
    i = np.where(whole, (top >> (np.uint64(20) - s)).astype(np.int64), 0)
    return i, np.where(whole, g, u)


@pytest.mark.parametrize("kind", ["uniform", "small", "below", "above", "nodes", "tiny"])
def test_split_floor_is_exact(kind):
    rng = np.random.default_rng(3)
    n = 200000
    nodes = rng.integers(0, 4096, n).astype(np.float64)
    u = {"uniform": lambda: rng.uniform(0, 4096, n), "small": lambda: rng.uniform(0, 2, n),
         "below": lambda: np.nextafter(nodes + 1, 0.0), "above": lambda: np.nextafter(nodes, 5000.0),
         "nodes": lambda: nodes, "tiny": lambda: np.ldexp(rng.uniform(0.5, 1, n), -rng.integers(0, 1070, n))}[kind]()
    u = u[(u >= 0) & (u < 4096)]
    i, f = split_floor(u)
    assert np.array_equal(i, np.floor(u).astype(np.int64))
    assert np.array_equal(f, u - np.floor(u))
