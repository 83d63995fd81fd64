"""Loading, keys and ordering of the particle state: positions on and outside the faces of the box, any
number of sub-cell bits, with and without the short-range force.  The caller's order is arbitrary, so the
accelerations of wrapped and unwrapped positions are the same bits; FP32 against FP64 mode: 1e-5 relative
RMS, the FP32 bar (the sets have no close pairs)."""

import numpy as np
import pytest

import p3m_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mesh,sub_bits", [(1, 20, 3), (33, 20, 0), (5003, 24, 3), (4096, 24, 2), (8193, 32, 5)])
@pytest.mark.parametrize("short_range", [True, False])
def test_positions_outside_the_box(n, mesh, sub_bits, short_range):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, P3MError, build
    build.build()
    box = 50.0
    x = np.mod(S.uniform_random(n, box, 7 + n), box)
    x = np.round(x * 64) / 64  # exact under shifts by the box
    x[0, 0] = 0.0
    y = x + box * np.random.default_rng(n).integers(-2, 3, x.shape)
    y[0, 0] = -0.0 if n % 2 else box
    got = {}
    for precision in ("mixed", "fp64"):
        with P3M(box, n, mesh, softening=0.3, sub_bits=sub_bits, short_range=short_range, precision=precision) as sim:
            for name, p in (("in", x), ("out", y)):
                sim.set_particles(p, np.zeros_like(p), a=1.0)
                got[precision, name] = sim.forces(1.0)
            with pytest.raises(P3MError):
                bad = x.copy()
                bad[1, n // 2] = np.nan
                sim.set_particles(bad, np.zeros_like(p), a=1.0)
        assert np.array_equal(got[precision, "in"], got[precision, "out"])
    a, b = got["mixed", "in"], got["fp64", "in"]
    scale = np.sqrt((b ** 2).sum())
    if n > 1:
        assert np.sqrt(((a - b) ** 2).sum()) <= 1e-5 * scale


@pytest.mark.parametrize("n,mesh", [(1, 20), (1023, 48), (1024, 48), (1025, 48), (4097, 64), (262143, 192), (262144, 192),
                                    (262145, 192), (270337, 192)])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_sort_at_tile_edges(n, mesh, precision):
    """The sort at the edges of its tiles and of its two methods: every particle is found by its neighbours
    (the number of pairs within the cutoff, against a k-d tree; at most two pairs lie within the FP32 mode's
    coordinate rounding of the cutoff) and again after a second sort of the sorted state."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spatial = pytest.importorskip("scipy.spatial")
    from paper_1510_07621_gb300 import P3M, build
    build.build()
    box = 100.0
    x = np.mod(S.uniform_random(n, box, 11 + n), box)
    tree = spatial.cKDTree(x.T, boxsize=box)
    rc = 4.5 * 1.25 * box / mesh
    want = int(tree.count_neighbors(tree, rc)) - n
    with P3M(box, n, mesh, softening=0.3, precision=precision) as sim:
        sim.set_particles(x, np.zeros_like(x), a=1.0)
        first = sim.forces(1.0)
        for _ in range(2):
            assert abs(sim.diagnostics()["pairs"] - want) <= (4 if precision == "mixed" else 0)
            again = sim.forces(1.0)
        assert np.array_equal(first, again)


@pytest.mark.parametrize("n", [5003, 900001, 3000001])
@pytest.mark.parametrize("where", ["device", "pinned", "pageable"])
def test_results_in_the_callers_order(n, where):
    """Positions and momenta come back as they were given after a sort, whichever way they take (written in
    place or through the inverse permutation, by size), and the accelerations do not depend on what else is
    asked for."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, build
    build.build()
    gen = torch.Generator().manual_seed(n)
    pos = torch.rand((3, n), generator=gen, dtype=torch.float64) * 100.0
    mom = torch.randn((3, n), generator=gen, dtype=torch.float64)

    def array():
        a = torch.zeros((3, n), dtype=torch.float64)
        return a.cuda() if where == "device" else a.pin_memory() if where == "pinned" else a

    with P3M(100.0, n, 64, short_range=False) as sim:
        sim.set_particles(pos, mom, a=1.0)
        alone = array()
        sim.forces(1.0, out=alone)
        p, m, a, only = array(), array(), array(), array()
        sim.get_particles(p, m, a)
        sim.get_particles(None, only)
        torch.cuda.synchronize()
    assert torch.equal(p.cpu(), pos) and torch.equal(m.cpu(), mom) and torch.equal(only.cpu(), mom)
    assert torch.equal(a.cpu(), alone.cpu())


def test_sort_timeout_with_many_particles():
    """The injected sort timeout also reaches a context whose sort has no look-back of its own (more than 2^18
    particles): P3M_ETIMEOUT, unchanged positions, and the same forces once the injection is cleared."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, P3MError, _lib, build
    build.build()
    lib = _lib.load()
    n, box = 300007, 100.0
    x = np.mod(S.uniform_random(n, box, 23), box)
    with P3M(box, n, 64, short_range=False) as sim:
        sim.set_particles(x, np.zeros_like(x), a=1.0)
        first = sim.forces(1.0)
        sim.set_particles(x, np.zeros_like(x), a=1.0)
        assert lib.p3m_inject_fault(sim._ctx, _lib.P3M_INJECT_SORT_TIMEOUT, 2000) == _lib.P3M_OK
        with pytest.raises(P3MError) as e:
            sim.forces(1.0)
        assert e.value.code == _lib.P3M_ETIMEOUT
        assert np.array_equal(sim.get_particles()[0], x)
        assert lib.p3m_inject_fault(sim._ctx, _lib.P3M_INJECT_NONE, 0) == _lib.P3M_OK
        assert np.array_equal(sim.forces(1.0), first)
