"""Every list kernel of the FP32 pair force and of its VJP (lists shared by 4, 8 or 16 particles, evaluated every
160 or 96 entries, both forms of the factor) where it can go wrong: a work item and a list with one particle more
or less, rows that wrap, a short and a long cutoff, coincident particles.  The lists' sizes are selected, since
small sets would take lists of 4.  Bars: those of the pair lists' own tests, 1e-5 relative RMS of the oracle for
the short-range force, 2e-5 for the VJP, and the oracle's pairs but for those within 1e-6 of the cutoff."""

import functools
import math

import numpy as np
import pytest

import p3m_synth as S
from oracle import p3m_oracle as O

pytestmark = pytest.mark.gpu

BOX = 50.0
KERNELS = [(4, 5), (8, 5), (16, 5), (16, 3)]


@pytest.fixture(scope="module")
def mod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import build
    build.build()
    import paper_1510_07621_gb300 as m
    from paper_1510_07621_gb300 import _lib
    return m, _lib


@functools.lru_cache(maxsize=None)
def _case(kind, n, mesh, cutoff, softening):
    x = S.uniform_random(n, BOX, 4000 + n + mesh)
    if kind == "cell":  # half of them inside one small region of one cell
        m = n // 2
        x[:, :m] = 0.45 * BOX + 0.02 * BOX * S.uniform_random(m, 1.0, 4001 + n)
    elif kind == "corner":  # half of them around the box's corner, in eight cells and all images
        m = n // 2
        x[:, :m] = 0.04 * BOX * (S.uniform_random(m, 1.0, 4001 + n) - 0.5)
    elif kind == "twins":
        x[:, 1::7] = x[:, ::7][:, :x[:, 1::7].shape[1]]
    x = np.mod(x, BOX)
    v = S.gaussian(19, 3 * n).reshape(3, n)
    p = O.Params(BOX, n, mesh, 1.25, cutoff, softening)
    ref, pairs = O.sr_accel(O.wrap(x, BOX), p)
    return x, v, ref, pairs, O.sr_vjp(O.wrap(x, BOX), v, p) + O.pm_vjp(O.wrap(x, BOX), v, p)


def _run(mod, x, v, mesh, cutoff, softening, kernel):
    m, _lib = mod
    with m.P3M(BOX, x.shape[1], mesh, 1.25, cutoff, softening=softening) as sim:
        assert sim._lib.p3m_inject_fault(sim._ctx, _lib.P3M_INJECT_PAIR_LISTS, 16 * kernel[0] + kernel[1]) == _lib.P3M_OK
        sim.set_particles(x, np.zeros_like(x), a=1.0)
        _, sr = sim.forces_split()
        return sr, sim.diagnostics()["pairs"], sim.force_vjp(v)


@pytest.mark.parametrize("kind,n,mesh,cutoff,softening", [
    ("cell", 30, 20, 4.5, 0.0), ("cell", 32, 26, 4.5, 0.02), ("cell", 34, 32, 4.5, 0.5), ("cell", 62, 20, 4.5, 0.02),
    ("cell", 66, 32, 4.5, 0.02), ("cell", 190, 26, 4.5, 0.02), ("cell", 192, 26, 4.5, 0.5), ("cell", 194, 26, 4.5, 0.02),
    ("corner", 318, 26, 4.5, 0.02), ("corner", 320, 26, 4.5, 0.5), ("corner", 322, 26, 4.5, 0.02),
    ("corner", 1500, 20, 4.5, 0.02), ("cell", 1500, 24, 4.5, 0.3), ("twins", 700, 26, 4.5, 0.02),
    ("twins", 700, 24, 4.5, 0.5), ("uniform", 4097, 24, 1.5, 0.02), ("uniform", 4097, 24, 2.0, 0.02),
    ("uniform", 4097, 48, 6.0, 0.02), ("uniform", 4097, 48, 6.0, 1.0),
])
@pytest.mark.parametrize("kernel", KERNELS)
def test_list_kernels(mod, kernel, kind, n, mesh, cutoff, softening):
    x, v, ref, pairs, vjp = _case(kind, n, mesh, cutoff, softening)
    sr, got, gv = _run(mod, x, v, mesh, cutoff, softening, kernel)
    assert math.sqrt(float(np.sum((sr - ref) ** 2))) <= 1e-5 * math.sqrt(float(np.sum(ref ** 2)))
    assert math.sqrt(float(np.sum((gv - vjp) ** 2))) <= 2e-5 * math.sqrt(float(np.sum(vjp ** 2)))
    rc, near = cutoff * 1.25 * BOX / mesh, 0
    for i in range(n):
        d = x[:, i + 1:] - x[:, i:i + 1]
        d -= BOX * np.round(d / BOX)
        near += 2 * int((np.abs(np.sqrt((d ** 2).sum(0)) - rc) < 1e-6 * rc).sum())
    assert abs(got - pairs) <= near


def test_each_size_has_its_kernel(mod):
    """Lists of another size add in another order: the bits differ, in force and (but for the length) in VJP."""
    x, v, *_ = _case("corner", 1500, 20, 4.5, 0.02)
    got = [_run(mod, x, v, 20, 4.5, 0.02, k) for k in KERNELS]
    for a in range(len(KERNELS)):
        for b in range(a):
            assert not np.array_equal(got[a][0], got[b][0])
            assert np.array_equal(got[a][2], got[b][2]) == (KERNELS[a][0] == KERNELS[b][0])


def test_sizes_that_no_kernel_has(mod):
    m, _lib = mod
    with m.P3M(BOX, 1000, 20) as sim:
        for arg in (0, 4, 16 * 5 + 5, 16 * 32 + 5, -1, 16 * 16 + 4):
            assert sim._lib.p3m_inject_fault(sim._ctx, _lib.P3M_INJECT_PAIR_LISTS, arg) == _lib.P3M_EINVAL
    assert m._lib.load().p3m_inject_fault(None, _lib.P3M_INJECT_PAIR_LISTS, 16 * 16 + 5) == _lib.P3M_EINVAL
