"""Small lattices where only a smaller cluster can be had than the one their rounds ask for, down to a single CTA and
to none that holds a round's attempts, when rounds are launched one by one: the replay's lattices in every case."""
import numpy as np
import pytest

import cpm_workloads as cw
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# name, workload, active blocks (two rounds or more per sub-pass), whether it moves and is tracked
CASES = [
    ("2d_144", lambda: cw.random_small(560, dim=2, n=48, n_cells=20, edge=3, act=True, obstacles=0.04, a=4, P=2), 144),
    ("2d_256", lambda: cw.random_small(561, dim=2, n=64, n_cells=20, edge=3, obstacles=0.04, a=4, P=2), 256),
    ("2d_289", lambda: cw.random_small(562, dim=2, n=68, n_cells=40, edge=3, act=True, a=4, P=2), 289),
    ("3d_512", lambda: cw.random_small(563, dim=3, n=32, n_cells=40, edge=3, act=True, n_types=3, a=4, P=4), 512),
    ("3d_4096", lambda: cw.random_small(564, dim=3, n=64, n_cells=200, edge=4, a=4, P=4), 4096),
    ("2d_moving_729", lambda: cw.with_motility(
        cw.random_small(565, dim=2, n=108, n_cells=40, edge=4, a=4, P=1), chem=cw.circular_field(108, 108, 1, 2),
        lambda_chem=15, lambda_pers=10, mu=0.5, dt=2), 729),
]


@pytest.mark.parametrize("name,factory,n_active", CASES, ids=[c[0] for c in CASES])
def test_smaller_clusters_give_the_same_lattice(name, factory, n_active):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    w = factory()
    rounds = w.a ** w.dim                     # of an MCS
    ref, sims = oracle.State(w, track=w.pers_on), {k: cpm.Sim(w) for k in (16, 11, 8, 4, 2, 1)}
    for k, sim in sims.items():
        sim.limit_cluster(k)
        if w.pers_on:
            sim.track_centroids(True)
    for step in (1, 2):
        ref.replay_run(step)
        for k, sim in sims.items():
            before = sim.launches()
            sim.step(step)
            launches = sim.launches() - before
            largest = 1 << (k.bit_length() - 1)
            if n_active <= 256 * largest:
                assert launches <= 6 * step, k    # a span, and what follows an MCS of moving, tracked cells
            else:
                assert launches >= rounds * step, k
            V, A = sim.read_tallies()
            assert np.array_equal(sim.read_lattice(), ref.lattice), k
            assert np.array_equal(V, ref.V) and np.array_equal(A, ref.A), k
            if ref.act is not None:
                assert np.array_equal(sim.read_act(), ref.act), k
            if w.pers_on:
                assert np.array_equal(sim.read_persistence(), ref.pers_dir), k
                assert np.array_equal(sim.read_centroid_sums(), ref.csum), k
    for ctas in (0, 17, -1):
        with pytest.raises(cpm.CPMError):
            sims[1].limit_cluster(ctas)
    for sim in sims.values():
        sim.close()
