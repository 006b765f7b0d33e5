"""A launch that runs many MCS of a batch of small lattices is bounded by the rounds of its longest member."""
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


def test_a_launch_is_bounded_by_its_rounds(cpm):
    w = cw.random_small(530, dim=2, n=40, n_cells=6, edge=5, act=True, a=40, c=2, P=1)
    v = cw.random_small(531, dim=2, n=16, n_cells=4, edge=3, act=True, a=4, c=2, P=1)
    batch, refs = cpm.Batch([v, w]), [oracle.State(v), oracle.State(w)]
    before = batch.launches()
    batch.step(70)
    launches = batch.launches() - before
    for k, ref in enumerate(refs):
        ref.replay_run(70)
        assert np.array_equal(batch.read_lattice(k), ref.lattice), k
    assert 70 * 1600 / 32768 <= launches <= 70  # 1,600 rounds per MCS of the longest member
    batch.close()
