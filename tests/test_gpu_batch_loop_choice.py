"""The autotuner of a batch of small lattices, whose steps are one launch, times the launches per round that its
bricks shape; the steps before and after it are those of the replay."""
import numpy as np
import pytest

import cpm_workloads as cw
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cpm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import build as B
    B.build()
    from paper_2312_09317_gb300 import cpm as c
    c.load()
    return c


@pytest.mark.parametrize("dim,n,candidates", [(2, 16, 6), (3, 8, 7)])
def test_autotune_times_a_launch_per_round(cpm, dim, n, candidates):
    ws = [cw.random_small(520 + k, dim=dim, n=n, n_cells=5, edge=3, act=True, a=4, P=1) for k in range(3)]
    batch, refs = cpm.Batch(ws), [oracle.State(w) for w in ws]
    rounds = ws[0].a ** dim                   # per MCS
    mcs = candidates * 3                      # one warm-up and two timed ones each
    before = batch.launches()
    assert 0 <= batch.autotune(2) < candidates
    assert batch.launches() - before >= mcs * rounds
    before = batch.launches()
    batch.step(3)
    assert batch.launches() - before == 1     # and a step is one launch again
    for k, ref in enumerate(refs):
        ref.replay_run(mcs + 3)
        assert np.array_equal(batch.read_lattice(k), ref.lattice), k
    batch.close()
