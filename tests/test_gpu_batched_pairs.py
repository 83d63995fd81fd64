"""The batched pair launch over several simulations: which of them it takes (its own two launches per step stand
in for the pair kernel's one, so a member's launches count them), and that every member's trajectory and pair
count equal those of its individual run bit for bit, also where members differ in list size, in list length or
in the factor's form, and after a member's tuning changes."""

import numpy as np
import pytest

import p3m_synth as S

pytestmark = pytest.mark.gpu

A = S.log_spaced_steps(0.05, 0.1, 6)


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


def _open(mod, spec):
    """spec: particles per side, seed, softening, list group (0: by the particle number), list length"""
    m, _lib = mod
    n_p, seed, soft, group, blocks = spec
    sim = m.P3M(60.0, n_p ** 3, max(20, n_p + n_p % 2), softening=soft, stream=0)
    pos, mom = S.zeldovich(n_p, 60.0, A[0], seed)
    sim.set_particles(pos, mom, a=A[0])
    _lets(mod, sim, group, blocks)
    return sim


def _lets(mod, sim, group, blocks):
    m, _lib = mod
    assert sim._lib.p3m_inject_fault(sim._ctx, _lib.P3M_INJECT_PAIR_LISTS, 16 * group + blocks) == _lib.P3M_OK


def _alone(mod, spec, a):
    with _open(mod, spec) as sim:
        for k in range(len(a) - 1):
            sim.step(a[k], a[k + 1] - a[k])
        d = sim.diagnostics()
        return sim.get_particles() + (d["pairs"], d["launches"])


# list sizes forced on small sets, each among members that do not qualify
SETS = {
    4: [(16, 1, 0.02, 4, 5), (20, 2, 0.02, 4, 3), (24, 3, 0.02, 4, 5), (27, 4, 0.02, 4, 5), (16, 5, 1.0, 4, 5)],
    8: [(24, 1, 0.02, 8, 5), (17, 2, 0.02, 4, 5), (28, 3, 0.02, 8, 3), (31, 4, 0.02, 8, 5)],
    16: [(40, 1, 0.02, 16, 5), (24, 2, 0.02, 16, 3), (21, 3, 0.02, 16, 5), (36, 4, 0.02, 16, 5), (17, 5, 0.02, 4, 5)],
}


def _qualifies(group, spec):
    return spec[2] < 0.5 and spec[3] == group and (group != 16 or spec[4] == 5)


@pytest.mark.parametrize("use_graph", [False, True])
@pytest.mark.parametrize("group", [4, 8, 16])
def test_members_equal_their_own_runs(mod, group, use_graph):
    m, _ = mod
    specs = SETS[group]
    takes = [_qualifies(group, s) for s in specs]
    assert sum(takes) >= 3 and not all(takes)
    alone = [_alone(mod, s, A) for s in specs]
    sims = [_open(mod, s) for s in specs]
    with m.Ensemble(sims, batched=True) as ens:
        ens.run(A, use_graph=use_graph)
    for sim, took, (pos, mom, pairs, launches) in zip(sims, takes, alone):
        d, (gp, gm) = sim.diagnostics(), sim.get_particles()
        assert np.array_equal(gp, pos) and np.array_equal(gm, mom)
        assert d["pairs"] == pairs
        if not use_graph:
            assert d["launches"] == launches + (len(A) - 1 if took else 0)
        sim.close()


@pytest.mark.parametrize("use_graph", [False, True])
def test_a_member_tuned_later(mod, use_graph):
    """A member's lists change between two runs of one ensemble: it leaves the batched launch."""
    m, _ = mod
    specs = [(24, 7, 0.02, 16, 5), (21, 8, 0.02, 16, 5), (28, 9, 0.02, 16, 5)]
    want = []
    for k, s in enumerate(specs):
        with _open(mod, s) as sim:
            sim.run_steps(A[:3], use_graph=False)
            if k == 1:
                _lets(mod, sim, 16, 3)
            sim.run_steps(A[2:], use_graph=False)
            want.append(sim.get_particles())
    sims = [_open(mod, s) for s in specs]
    with m.Ensemble(sims, batched=True) as ens:
        ens.run(A[:3], use_graph=use_graph)
        _lets(mod, sims[1], 16, 3)
        ens.run(A[2:], use_graph=use_graph)
    for sim, (pos, mom) in zip(sims, want):
        gp, gm = sim.get_particles()
        assert np.array_equal(gp, pos) and np.array_equal(gm, mom)
        sim.close()
