"""Which pairs the FP32 mode lets interact, on whole sets, component by component.

A set with at least as many particles as chaining cells decides r < r_c by the FP32 r^2 of the
cell-relative coordinates (x_j against x_i shifted into j's cell), emulated here bit for bit; about one
pair in 10^7 lies where FP32 does not resolve its side, so the sets are given thousands.  Bars: the same
number of ordered pairs, and every component of the short-range force and of the force VJP within 1e-4 of
that field's rms value of the FP64 sum over those pairs: five times the largest FP32 rounding of a
component (1.8e-5 emulated, on such sets).  One pair on the other side changes the force by 5e-4 or more, and
the VJP of the sets softened by 1.5 spacings by 1e-3 (close pairs dominate it otherwise)."""

import math

import numpy as np
import pytest

import p3m_synth as S
from oracle import p3m_oracle as O

pytestmark = pytest.mark.gpu

R_S, SUB_BITS = 1.25, 3


def _directed(x, box, r):
    """All ordered pairs closer than r: i, j and d = x_j - x_i (minimum image)."""
    tree = pytest.importorskip("scipy.spatial").cKDTree(x.T, boxsize=box)
    p = tree.query_pairs(r, output_type="ndarray").T
    i, j = np.concatenate([p, p[::-1]], axis=1)
    d = x[:, j] - x[:, i]
    return i, j, d - box * np.round(d / box)


def _fp32_inside(x, i, j, box, rc):
    """r < r_c as the FP32 mode decides it."""
    f4 = np.float32
    nc = int(np.floor(box / rc))
    cs, nf = box / nc, nc << SUB_BITS
    c = np.minimum((x * (nf / box)).astype(np.int64), nf - 1) >> SUB_BITS
    rel = (x - c * cs).astype(f4)
    r2 = np.full(i.size, 1e-20, f4)
    for d in range(3):
        step = c[d, j] - c[d, i]
        image = np.where(step > 1, -box, np.where(step < -1, box, 0.0))
        s = (c[d, j] * cs + image) - c[d, i] * cs
        hi = s.astype(f4)
        t = rel[d, j] - ((rel[d, i] - hi) - (s - hi).astype(f4))
        # an FMA: the FP64 product of two FP32 values is exact, the sum's double rounding is 2^-29 rare
        r2 = (t.astype(np.float64) ** 2 + r2).astype(f4)
    return r2 < f4(rc * rc)


def _pair_sums(x, v, box, mesh, cutoff, softening):
    """Ordered pairs, short-range accelerations and force VJP with the FP32 mode's decisions."""
    erfc = pytest.importorskip("scipy.special").erfc
    n = x.shape[1]
    rs = R_S * (box / mesh)
    rc, eps = cutoff * rs, softening * box / n ** (1.0 / 3.0)
    gm = 3.0 * box ** 3 / (8.0 * math.pi * n)
    i, j, d = _directed(x, box, rc * (1 + 1e-5))
    r2 = (d * d).sum(0)
    ok = np.where(np.abs(r2 / rc ** 2 - 1) < 1e-5, _fp32_inside(x, i, j, box, rc), r2 < rc * rc)
    i, j, d, r2 = i[ok], j[ok], d[:, ok], r2[ok]
    u = 0.5 * np.sqrt(r2) / rs
    g = erfc(u) + 2.0 / math.sqrt(math.pi) * u * np.exp(-u * u)
    s2 = 1.0 / (r2 + eps * eps)
    h = g * s2 ** 1.5
    hr = -(np.sqrt(r2) / rs ** 3) * np.exp(-u * u) / (2 * math.sqrt(math.pi)) * s2 ** 1.5 - 3.0 * h * s2
    w = v[:, j] - v[:, i]
    vj = h * w + hr * (d * w).sum(0) * d
    acc, vjp = np.zeros_like(x), np.zeros_like(x)
    for e in range(3):
        acc[e] = gm * np.bincount(i, h * d[e], n)
        vjp[e] = gm * np.bincount(i, vj[e], n)
    return i.size, acc, vjp


def _at_the_cutoff(x, box, rc, seed):
    """Moves particles so that many disjoint pairs lie within 2e-7 of the cutoff; returns how many."""
    i, j, d = _directed(x, box, rc * 1.02)
    r = np.sqrt((d * d).sum(0))
    near = np.flatnonzero((r > 0.98 * rc) & (i < j))
    rng = np.random.default_rng(seed)
    used, moved = np.zeros(x.shape[1], bool), 0
    for k in rng.permutation(near):
        a, b = i[k], j[k]
        if used[a] or used[b]:
            continue
        used[a] = used[b] = True
        x[:, b] = x[:, a] + d[:, k] * (rc * (1 + rng.uniform(-2e-7, 2e-7)) / r[k])
        moved += 1
    return np.mod(x, box), moved


def _check(x, v, box, mesh, cutoff, softening):
    from paper_1510_07621_gb300 import P3M
    pairs, acc, vjp = _pair_sums(x, v, box, mesh, cutoff, softening)
    p = O.Params(box, x.shape[1], mesh, R_S, cutoff, softening)
    with P3M(box, x.shape[1], mesh, R_S, cutoff, softening=softening) as sim:
        sim.set_particles(x, np.zeros_like(x), a=1.0)
        _, sr = sim.forces_split()
        assert sim.diagnostics()["pairs"] == pairs
        got = sim.force_vjp(v) - O.pm_vjp(x, v, p)
    assert np.abs(sr - acc).max() <= 1e-4 * math.sqrt(float(np.mean(acc ** 2)))
    assert np.abs(got - vjp).max() <= 1e-4 * math.sqrt(float(np.mean(vjp ** 2)))


@pytest.mark.parametrize("n_p,mesh,cutoff,softening", [
    (16, 18, 4.5, 0.02), (16, 24, 4.5, 0.02), (16, 32, 4.5, 1.5), (24, 48, 4.5, 0.02), (24, 48, 4.5, 1.5),
    (36, 54, 4.5, 0.02), (36, 72, 4.5, 0.02), (24, 32, 3.0, 1.5),
])
def test_pairs_at_the_cutoff(n_p, mesh, cutoff, softening):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import build
    build.build()
    box = 1.5625 * n_p
    x, _ = S.zeldovich(n_p, box, 0.3, 600 + n_p + mesh)
    x, moved = _at_the_cutoff(np.mod(x, box), box, cutoff * R_S * box / mesh, mesh)
    assert moved > x.shape[1] // 8
    v = np.random.default_rng(mesh).normal(size=x.shape)
    _check(x, v, box, mesh, cutoff, softening)


def test_lattice_pairs_exactly_at_the_cutoff():
    """A lattice and cells that FP32 holds exactly, with 30 neighbours of each particle at r = r_c: none
    interacts, in the number of pairs and in the VJP (the force of a lattice is zero either way)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import build
    build.build()
    x = S.lattice(20, 20.0)
    v = np.random.default_rng(2).normal(size=x.shape)
    q = np.stack(np.meshgrid(*[np.arange(-5, 6)] * 3)).reshape(3, -1)
    inside = int(((q * q).sum(0) < 25).sum()) - 1
    pairs, _, vjp = _pair_sums(x, v, 20.0, 20, 4.0, 1.5)
    assert pairs == 8000 * inside
    from paper_1510_07621_gb300 import P3M
    with P3M(20.0, 8000, 20, R_S, 4.0, softening=1.5) as sim:
        sim.set_particles(x, np.zeros_like(x), a=1.0)
        sim.forces(1.0)
        assert sim.diagnostics()["pairs"] == pairs
        got = sim.force_vjp(v) - O.pm_vjp(x, v, O.Params(20.0, 8000, 20, R_S, 4.0, 1.5))
    assert np.abs(got - vjp).max() <= 1e-4 * math.sqrt(float(np.mean(vjp ** 2)))
