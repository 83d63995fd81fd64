"""The FP32 pair factor and its derivative at distances around a small softening, where most of a dense core's
pairs are: isolated pairs at 0.3 to 4 softenings against the FP64 mode.  A halo adds thousands of such pairs,
so the mean of the relative errors counts: at most 2e-7 for the force and 3e-7 for the VJP (relative to the sum
of its two terms), the FP32 rounding that has a sign (below 1e-7 and 2e-7) and five standard errors of the
mean over 729 pairs (the error of one pair has an rms value of 5e-7 or less, mostly its coordinates')."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eps_rs", [0.016, 0.024, 0.032, 0.033, 0.1])
@pytest.mark.parametrize("cutoff", [4.5, 3.0])
def test_pairs_around_the_softening(eps_rs, cutoff):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, build
    build.build()
    box, mesh = 100.0, 128 if cutoff == 4.5 else 86
    r_s = 1.25 * box / mesh
    k = int(box / (2.5 * cutoff * r_s))  # pairs on a lattice wide enough that only partners meet
    assert k >= 9
    k = 9
    m, n = k ** 3, 2 * k ** 3
    eps = eps_rs * r_s
    rng = np.random.default_rng(int(1e4 * eps_rs))
    at = (np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij")).reshape(3, -1) + 0.5) * (box / k)
    u = rng.normal(size=(3, m))
    u /= np.sqrt((u ** 2).sum(0))
    r = 0.3 * eps * (4.0 / 0.3) ** rng.uniform(size=m)
    x = np.concatenate([at, at + r * u], axis=1)
    v = np.concatenate([np.zeros_like(u), u], axis=1)
    got = {}
    for precision in ("mixed", "fp64"):
        with P3M(box, n, mesh, 1.25, cutoff, softening=eps * n ** (1.0 / 3.0) / box, precision=precision) as sim:
            sim.set_particles(x, np.zeros_like(x), a=1.0)
            _, sr = sim.forces_split()
            vjp = sim.force_vjp(v) - sim.force_vjp(np.zeros_like(v))
            got[precision] = ((sr[:, :m] * u).sum(0), (vjp[:, :m] * u).sum(0))
    (fa, va), (fb, vb) = got["mixed"], got["fp64"]
    assert abs(float(np.mean(fa / fb - 1.0))) <= 2e-7
    # h and the other term, (h'/r) r^2 = -3 h r^2 / (r^2 + eps^2) to 1e-4 at these distances
    h = fb / r
    scale = h * (1.0 + 3.0 * r * r / (r * r + eps * eps))
    assert abs(float(np.mean((va - vb) / scale))) <= 3e-7
