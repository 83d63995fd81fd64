"""The autotuner times list lengths only where a kernel has two of them (lists shared by 16 particles): elsewhere
it would time one kernel twice and keep a length by noise."""

import numpy as np
import pytest

import p3m_synth as S

pytestmark = pytest.mark.gpu


def test_list_length_of_small_lists_stays():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_07621_gb300 import P3M, _lib, build
    build.build()
    x = S.uniform_random(4096, 50.0, 3)
    launches = {}
    for group in (4, 8, 16):
        for blocks in (3, 5):
            with P3M(50.0, 4096, 24) as sim:
                sim.set_particles(x, np.zeros_like(x), a=1.0)
                assert sim._lib.p3m_inject_fault(sim._ctx, _lib.P3M_INJECT_PAIR_LISTS, 16 * group + blocks) == _lib.P3M_OK
                sim.autotune()
                launches[group, blocks] = sim.diagnostics()["launches"]
                if group < 16:
                    assert sim.tuning()["tile_blocks"] == blocks
    # (sub_bits change the number of sort passes, but are all timed alike)
    assert max(launches[4, b] for b in (3, 5)) < min(launches[16, b] for b in (3, 5))
    assert max(launches[8, b] for b in (3, 5)) < min(launches[16, b] for b in (3, 5))
