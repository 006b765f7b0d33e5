"""Batches that mix members with and without the Act term, on each of the batch's loops.

The words of a member with Act carry stamps, which are clamped every 64 MCS; those of a member without are plain
ids and have to stay so.  A plain word reads as stamp 0, whose age passes 128 at MCS 192 and a stamp's period at 256,
so the members run past both, bit for bit against the replay oracle and, as read, in the range of ids.
"""
import numpy as np
import pytest

import cpm_workloads as cw
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["cta", "track", "loop"])
@pytest.mark.parametrize("dim,n", [(2, 16), (3, 8)])
def test_members_without_act_keep_plain_ids(dim, n, mode):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    ws = [cw.random_small(500 + k, dim=dim, n=n, n_cells=6, edge=3, obstacles=0.04, act=k % 2 == 0, a=4, P=1)
          for k in range(4)]
    batch, refs = cpm.Batch(ws), [oracle.State(w) for w in ws]
    batch.set_persistent(mode == "loop")
    batch.track_centroids(mode == "track")
    for step in (191, 2, 66, 70):
        batch.step(step)
        for k, ref in enumerate(refs):
            ref.replay_run(step)
            on_device = torch.empty(ref.lattice.shape, dtype=torch.int32, device="cuda")
            batch.read_lattice(k, on_device)
            V, A = batch.read_tallies(k)
            assert np.array_equal(batch.read_lattice(k), ref.lattice), (k, ref.t)
            assert np.array_equal(on_device.cpu().numpy(), ref.lattice), (k, ref.t)
            assert np.array_equal(V, ref.V) and np.array_equal(A, ref.A), (k, ref.t)
            if ref.act is not None:
                assert np.array_equal(batch.read_act(k), ref.act), (k, ref.t)
    batch.close()
