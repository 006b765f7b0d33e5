"""Lattices on both sides of the sizes where cpm_step changes its route, against the replay oracle, bit for bit.

A lattice with at most 4,096 active blocks per round runs many rounds per launch on one cluster of CTAs
(with at most 128 of them and a lattice that fits, in one CTA's shared memory), a larger one a launch per
round.  The cases sit at the edges: one active block, the last resident size and the first that is not,
a lattice too large for shared memory, 4,096 active blocks and the next size, a block edge that is not a
power of two, and odd numbers of rounds per call, so that either tally buffer is the current one.
"""
import numpy as np
import pytest

import cpm_workloads as cw
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _small(seed, dim, n, cells, **kw):
    return cw.random_small(seed, dim=dim, n=n, n_cells=cells, edge=3, obstacles=0.04, **kw)


def _wide(seed, dim, n):
    w = _small(seed, dim, n, 24, act=True, n_types=2, a=4, P=1, T=1500.0)
    return w.replace(J=w.J * 100, lambda_v=w.lambda_v * 40, lambda_p=w.lambda_p * 30, lambda_act=w.lambda_act * 20011)


CASES = [
    # (name, workload, sub-passes of the calls)
    ("2d_one_block", lambda: _small(61, 2, 8, 3, act=True, a=8, P=16), (3, 70)),
    ("2d_resident_121", lambda: _small(62, 2, 44, 20, act=True, a=4, P=1), (1, 9)),
    ("2d_resident_s3", lambda: _small(63, 2, 48, 20, a=6, P=3), (5, 13)),
    ("2d_cluster_144", lambda: _small(64, 2, 48, 20, act=True, n_types=3, a=4, P=2), (3, 9)),
    ("2d_too_large_for_smem", lambda: _small(65, 2, 240, 90, act=True, a=60, P=900), (7, 90)),
    ("2d_4096", lambda: _small(66, 2, 256, 300, act=True, a=4, P=1), (1, 7)),
    ("2d_4225", lambda: _small(67, 2, 260, 300, act=True, a=4, P=1), (1, 7)),
    ("3d_resident_64", lambda: _small(68, 3, 32, 30, act=True, a=8, P=64), (5, 40)),
    ("3d_cluster_s3", lambda: _small(69, 3, 30, 30, act=True, a=6, P=27), (5, 40)),
    ("3d_4096", lambda: _small(70, 3, 64, 200, n_types=2, a=4, P=8), (3, 8)),
    # weights beyond the 32-bit products of the round kernels (lambda_Act above 2^19)
    ("2d_wide", lambda: _wide(72, 2, 48), (3, 9)),
    ("3d_wide", lambda: _wide(73, 3, 32), (3, 9)),
    ("3d_4913", lambda: _small(71, 3, 68, 200, act=True, a=4, P=8), (3, 8)),
]


def test_batch_members_in_one_cta_each():
    """304 members of up to 484 active blocks run in one CTA each, two stripes of attempts per round, mixed with
    smaller ones; across the Act stamp clamp at MCS 64, and back and forth between the batch's three loops."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    ws = [_small(400 + k, 2, (88, 64, 20, 16)[k % 4], 24, act=k % 3 != 0, n_types=1 + k % 2, a=4, P=(1, 4)[k % 2])
          for k in range(304)]
    picked = (0, 1, 2, 3, 150, 301, 303)
    batch, refs = cpm.Batch(ws), {k: oracle.State(ws[k]) for k in picked}
    for step, mode in ((63, "cta"), (2, "cta"), (1, "loop"), (2, "track"), (3, "cta")):
        batch.set_persistent(mode == "loop")
        batch.track_centroids(mode == "track")
        batch.step(step)
        for k, ref in refs.items():
            ref.replay_run(step)
            V, A = batch.read_tallies(k)
            assert np.array_equal(batch.read_lattice(k), ref.lattice), (k, mode)
            assert np.array_equal(V, ref.V) and np.array_equal(A, ref.A), (k, mode)
            if ref.act is not None:
                assert np.array_equal(batch.read_act(k), ref.act), (k, mode)
            st = batch.stats(k)
            assert st["accepts"] == ref.accepts and st["mcs"] == ref.t
    batch.close()


@pytest.mark.parametrize("name,factory,calls", CASES, ids=[c[0] for c in CASES])
def test_route_matches_replay(name, factory, calls):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    w = factory()
    sim, ref = cpm.Sim(w), oracle.State(w)
    for n in calls:
        sim.step_subpasses(n)
        ref.replay_subpasses(n)
        V, A = sim.read_tallies()
        assert np.array_equal(sim.read_lattice(), ref.lattice)
        assert np.array_equal(V, ref.V) and np.array_equal(A, ref.A)
        if ref.act is not None:
            assert np.array_equal(sim.read_act(), ref.act)
        assert sim.stats()["accepts"] == ref.accepts
    sim.close()
