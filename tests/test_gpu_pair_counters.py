"""The pair kernels' work counters on a set with a dense cell: blocks wholly inside the cutoff are counted apart
from tested ones (FP32 mode), what is evaluated covers the accepted pairs, and batches of blocks that are all
culled (those of the dense cell, for groups elsewhere) are counted."""

import numpy as np
import pytest

import p3m_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,group,blocks", [("mixed", 4, 5), ("mixed", 8, 5), ("mixed", 16, 5), ("mixed", 16, 3),
                                                    ("fp64", 0, 5)])
def test_counters(precision, group, blocks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, _lib, build
    build.build()
    box, n = 50.0, 6001
    x = S.uniform_random(n, box, 5)
    x[:, :5000] = 0.51 * box + 0.005 * box * S.uniform_random(5000, 1.0, 6)
    with P3M(box, n, 32, precision=precision) as sim:
        assert sim._lib.p3m_inject_fault(sim._ctx, _lib.P3M_INJECT_PAIR_LISTS, 16 * group + blocks) == _lib.P3M_OK
        sim.set_particles(np.mod(x, box), np.zeros_like(x), a=1.0)
        sim.forces(1.0)
        d = sim.diagnostics()
    inside, tested, evaluated = d["pair_warp_j"]
    batches, empty = d["pair_tiles"]
    assert 32 * (inside + evaluated) + 32 * n >= d["pairs"]  # (rounded to steps of 32 per group)
    assert 0 < evaluated <= tested
    assert 0 < empty < batches and d["pair_blocks_culled"] >= 32 * empty
    if precision == "fp64":
        assert inside == 0
    else:  # the dense cell's own pairs: nearly all of its 156 blocks against its 5000 particles
        assert 32 * inside > 0.9 * 5000 ** 2
