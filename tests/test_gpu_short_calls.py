"""Calls of a few rounds on small lattices: as quick as their rounds, with a launch each, and the same lattices as
longer calls, which run in one launch, whichever way the sub-passes are cut into calls."""
import numpy as np
import pytest

import cpm_workloads as cw
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# name, workload, rounds of a sub-pass, sub-passes of a call that repays a launch for all of its rounds
CASES = [
    ("resident_25_blocks", lambda: cw.point_cells_2d(seed=1, n=200, n_cells=100, a=40, P=400), 1, 200),
    ("resident_16_blocks", lambda: cw.random_small(550, dim=2, n=64, n_cells=30, edge=5, act=True, a=16, P=64), 1, 40),
    ("resident_3d", lambda: cw.random_small(551, dim=3, n=32, n_cells=30, edge=4, act=True, a=8, P=64), 1, 100),
    ("cluster_3d", lambda: cw.random_small(552, dim=3, n=64, n_cells=60, edge=6, act=True, a=8, P=64), 1, 20),
]


@pytest.mark.parametrize("name,factory,k,long_call", CASES, ids=[c[0] for c in CASES])
def test_a_call_launches_what_suits_its_rounds(name, factory, k, long_call):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    w = factory()
    sim, ref = cpm.Sim(w), oracle.State(w)
    for n in (1, 3, long_call, 2):
        before = sim.launches()
        sim.step_subpasses(n)
        launches = sim.launches() - before
        clamp = 1 if w.act_on and ref.t % 64 == 0 and ref.sp == 0 else 0
        assert launches == (1 if n == long_call else n * k + clamp), n
        ref.replay_subpasses(n)
        V, A = sim.read_tallies()
        assert np.array_equal(sim.read_lattice(), ref.lattice), n
        assert np.array_equal(V, ref.V) and np.array_equal(A, ref.A), n
        if ref.act is not None:
            assert np.array_equal(sim.read_act(), ref.act), n
        assert sim.stats()["accepts"] == ref.accepts
    sim.close()
