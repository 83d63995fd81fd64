"""The pair kernels' lists.

FP32: at the sizes where they can go wrong: groups of 16 particles with
one more or one less, cells around a whole work item, rows of cells that wrap, lists longer than one
chunk and one FP64 flush, both forms of the split factor (a softening small or large against r_s, a
short and a long cutoff) and both list lengths.  Bars: the short-range accelerations within 1e-5
relative RMS of the oracle (the FP32 bar), and the accepted pairs within the pairs whose distance
lies within 1e-6 of the cutoff.

FP64: groups of 8 particles with one more or one less, more candidate blocks than one round of masks
holds, and a table of the split factor that covers a short or a long range.  Bars: 1e-12 relative RMS
(the FP64 bar) and the same number of pairs.

FP32 force VJP: the same lists with v, both forms of the factor's derivative, coincident particles
(which have w but no force).  Bar: 2e-5 relative RMS of the oracle, the FP32 bar of the force VJP."""

import math

import numpy as np
import pytest

import p3m_synth as S
from oracle import p3m_oracle as O

pytestmark = pytest.mark.gpu


def _set(kind, n, box, seed):
    x = S.uniform_random(n, box, seed)
    if kind == "cell":  # half of them inside one small region of one cell
        m = n // 2
        x[:, :m] = 0.45 * box + 0.02 * box * S.uniform_random(m, 1.0, seed + 1)
    return np.mod(x, box)


@pytest.mark.parametrize("kind,n,mesh,cutoff,softening", [
    ("uniform", 2, 20, 4.5, 0.02), ("cell", 30, 20, 4.5, 0.0), ("cell", 32, 26, 4.5, 0.02),
    ("cell", 34, 32, 4.5, 0.02), ("cell", 62, 20, 4.5, 0.5), ("cell", 66, 32, 4.5, 0.02),
    ("cell", 1500, 20, 4.5, 0.02), ("cell", 1500, 24, 4.5, 0.3), ("cell", 6001, 32, 4.5, 0.02),
    ("uniform", 4097, 24, 1.5, 0.02), ("uniform", 4097, 48, 6.0, 0.02), ("uniform", 4097, 48, 6.0, 1.0),
])
@pytest.mark.parametrize("tile_blocks", [5, 3])
def test_pair_lists(kind, n, mesh, cutoff, softening, tile_blocks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, build
    build.build()
    box = 50.0
    x = _set(kind, n, box, 1000 + n + mesh)
    p = O.Params(box, n, mesh, 1.25, cutoff, softening)
    ref, pairs = O.sr_accel(O.wrap(x, box), p)
    with P3M(box, n, mesh, 1.25, cutoff, softening=softening) as sim:
        sim.set_particles(x, np.zeros_like(x), a=1.0)
        if tile_blocks == 3:  # the autotuner times both lengths; which one it keeps does not matter
            sim.autotune()
        _, sr = sim.forces_split()
        got = sim.diagnostics()["pairs"]
    # (no pair within the cutoff: the force is exactly zero)
    assert math.sqrt(float(np.sum((sr - ref) ** 2))) <= 1e-5 * math.sqrt(float(np.sum(ref ** 2)))
    d = x[:, :, None] - x[:, None, :] if n <= 1500 else None
    if d is not None:
        d -= box * np.round(d / box)
        r = np.sqrt((d ** 2).sum(0))
        rc = cutoff * 1.25 * box / mesh
        near = int((np.abs(r - rc) < 1e-6 * rc).sum())
        assert abs(got - pairs) <= near
    else:
        assert abs(got - pairs) <= max(4, int(2e-6 * pairs))


@pytest.mark.parametrize("kind,n,mesh,cutoff,softening", [
    ("uniform", 2, 20, 4.5, 0.02), ("cell", 14, 20, 4.5, 0.0), ("cell", 16, 26, 4.5, 0.02),
    ("cell", 18, 20, 4.5, 0.5), ("cell", 1500, 20, 4.5, 0.02), ("cell", 6001, 32, 4.5, 0.0),
    ("uniform", 4097, 24, 1.5, 0.02), ("uniform", 4097, 48, 6.0, 1.0),
])
def test_pair_masks_fp64(kind, n, mesh, cutoff, softening):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, build
    build.build()
    box = 50.0
    x = _set(kind, n, box, 2000 + n + mesh)
    p = O.Params(box, n, mesh, 1.25, cutoff, softening)
    ref, pairs = O.sr_accel(O.wrap(x, box), p)
    with P3M(box, n, mesh, 1.25, cutoff, softening=softening, precision="fp64") as sim:
        sim.set_particles(x, np.zeros_like(x), a=1.0)
        _, sr = sim.forces_split()
        got = sim.diagnostics()["pairs"]
    assert math.sqrt(float(np.sum((sr - ref) ** 2))) <= 1e-12 * math.sqrt(float(np.sum(ref ** 2)))
    assert got == pairs


@pytest.mark.parametrize("kind,n,mesh,cutoff,softening", [
    ("cell", 30, 20, 4.5, 0.02), ("cell", 34, 32, 4.5, 0.5), ("cell", 700, 20, 4.5, 0.02),
    ("twins", 700, 26, 4.5, 0.02), ("twins", 700, 24, 4.5, 0.5), ("uniform", 1000, 24, 1.5, 0.02),
    ("uniform", 1000, 48, 6.0, 1.0),
])
def test_force_vjp_lists(kind, n, mesh, cutoff, softening):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, build
    build.build()
    box = 50.0
    x = _set("uniform" if kind == "twins" else kind, n, box, 3000 + n + mesh)
    if kind == "twins":
        x[:, 1::7] = x[:, ::7]
    v = S.gaussian(17, 3 * n).reshape(3, n)
    p = O.Params(box, n, mesh, 1.25, cutoff, softening)
    ref = O.sr_vjp(O.wrap(x, box), v, p)
    with P3M(box, n, mesh, 1.25, cutoff, softening=softening) as sim:
        sim.set_particles(x, np.zeros_like(x), a=1.0)
        got = sim.force_vjp(v)
    mesh_part = O.pm_vjp(O.wrap(x, box), v, p)
    err = got - mesh_part - ref
    assert math.sqrt(float(np.sum(err ** 2))) <= 2e-5 * math.sqrt(float(np.sum((ref + mesh_part) ** 2)))


@pytest.mark.parametrize("box,mesh,cutoff,softening", [
    (100.0, 48, 4.5, 0.02), (100.0, 64, 4.5, 0.02), (70.0, 54, 4.5, 0.5), (30.0, 24, 2.5, 0.0),
])
@pytest.mark.parametrize("off", [3e-8, 2e-7, 1e-5])
def test_cutoff_decided_exactly(box, mesh, cutoff, softening, off):
    """Isolated pairs closer to the cutoff than FP32 resolves (its r is 4e-8 off at one sigma), in any
    direction and across the box's faces: each is inside or outside as its FP64 distance says, in the
    force and in its derivative.  Bar: the FP32 rounding, 1e-4 of the largest value; a pair on the wrong
    side is off by all of its short-range force, and by more than 1e-3 of the largest derivative."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, build
    build.build()
    rng = np.random.default_rng(mesh)
    rc = cutoff * 1.25 * box / mesh
    k = int(box / (2.5 * rc))  # pairs on a lattice wide enough that only partners meet
    assert k >= 1
    at = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij")).reshape(3, -1) * (box / k)
    m = at.shape[1]
    u = rng.normal(size=(3, m))
    u /= np.sqrt((u ** 2).sum(0))
    side = np.where(np.arange(m) % 2 == 0, -1.0, 1.0)  # inside, outside
    mid = at + 0.1 * rc * rng.uniform(-1, 1, (3, m))
    half = 0.5 * rc * (1.0 + side * off) * u
    x = np.mod(np.concatenate([mid - half, mid + half], axis=1), box)
    v = rng.normal(size=x.shape)
    got = {}
    for precision in ("mixed", "fp64"):
        with P3M(box, 2 * m, mesh, 1.25, cutoff, softening=softening, precision=precision) as sim:
            sim.set_particles(x, np.zeros_like(x), a=1.0)
            _, sr = sim.forces_split()
            got[precision] = sr, sim.force_vjp(v), sim.diagnostics()["pairs"]
    assert got["mixed"][2] == got["fp64"][2] == 2 * int((side < 0).sum())
    for a, b in zip(got["mixed"][:2], got["fp64"][:2]):
        assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max()


@pytest.mark.parametrize("fraction", [0.499, 0.5, 0.51, 0.999, 1.0, 1.1])
@pytest.mark.parametrize("kind,softening", [("uniform", 0.02), ("cell", 0.3)])
def test_list_group_sizes(fraction, kind, softening):
    """Lists of 4, 8 and 16 particles on both sides of the particle numbers where they change (as fractions of
    16 particles per resident warp), against the FP64 kernel: 1e-5 relative RMS of the short-range force and
    2e-5 of the VJP, the FP32 bars, and the same pairs (their coordinates' rounding, 1e-9 of the cutoff, may
    move one in 10^8)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, build
    build.build()
    n = int(16 * 18 * torch.cuda.get_device_properties(0).multi_processor_count * fraction)
    box, mesh = 60.0, 40
    x = np.mod(S.uniform_random(n, box, 17), box)
    if kind == "cell":
        m = n // 40
        x[:, :m] = 0.45 * box + 0.02 * box * S.uniform_random(m, 1.0, 18)
    v = np.random.default_rng(1).normal(size=x.shape)
    got = {}
    for precision in ("mixed", "fp64"):
        with P3M(box, n, mesh, softening=softening, precision=precision) as sim:
            sim.set_particles(x, np.zeros_like(x), a=1.0)
            _, sr = sim.forces_split()
            got[precision] = sr, sim.diagnostics()["pairs"], sim.force_vjp(v)
    (a, na, va), (b, nb, vb) = got["mixed"], got["fp64"]
    assert abs(na - nb) <= max(4, 2e-8 * nb)
    assert math.sqrt(float(np.sum((a - b) ** 2))) <= 1e-5 * math.sqrt(float(np.sum(b ** 2)))
    assert math.sqrt(float(np.sum((va - vb) ** 2))) <= 2e-5 * math.sqrt(float(np.sum(vb ** 2)))


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("softening", [0.02, 1.0])
def test_ensemble_members_keep_their_group_size(batched, softening):
    """Simulations whose lists have 4, 8 and 16 particles, advanced together (the pair sums of those of one
    group size and the additive factor in one launch, or all of them alone) and alone: the same bits."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, Ensemble, build
    build.build()
    a = S.log_spaced_steps(0.05, 0.08, 3)
    sets = [(p, *S.zeldovich(p, 60.0, a[0], 5 + p)) for p in (17, 30, 40, 21)]
    alone = []
    for p, pos, mom in sets:
        with P3M(60.0, p ** 3, max(20, p + p % 2), softening=softening, stream=0) as sim:
            sim.set_particles(pos, mom, a=a[0])
            for k in range(3):
                sim.step(a[k], a[k + 1] - a[k])
            alone.append(sim.get_particles())
    sims = [P3M(60.0, p ** 3, max(20, p + p % 2), softening=softening, stream=0) for p, _, _ in sets]
    for sim, (_, pos, mom) in zip(sims, sets):
        sim.set_particles(pos, mom, a=a[0])
    with Ensemble(sims, batched=batched) as ens:
        ens.run(a)
    for sim, (pos, mom) in zip(sims, alone):
        got = sim.get_particles()
        assert np.array_equal(got[0], pos) and np.array_equal(got[1], mom)
        sim.close()
