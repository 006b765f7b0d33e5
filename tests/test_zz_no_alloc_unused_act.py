"""cpm_step_noalloc leaves max_act unread: it takes a configuration without the Act term whatever max_act holds, as
the replay does, up to the numbers at which a search for a power of two above it would not end."""
import ctypes

import numpy as np
import pytest

import cpm_workloads as cw
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(2, 16), (3, 8)])
@pytest.mark.parametrize("max_act", [128, (1 << 30) + 1, (1 << 31) - 1, -(1 << 31)])
def test_max_act_is_not_read_without_the_act_term(dim, n, max_act):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    w = cw.random_small(540 + dim, dim=dim, n=n, n_cells=6, edge=3, obstacles=0.03, a=4, P=2)
    st = oracle.State(w)
    keep = []
    cfg = cpm.make_config(w, keep)
    for t in range(1, cpm.MAX_TYPES):
        cfg.max_act[t] = max_act
    lat = torch.from_numpy(st.lattice.copy()).cuda()
    V, A = torch.from_numpy(st.V.copy()).cuda(), torch.from_numpy(st.A.copy()).cuda()
    ct = torch.from_numpy(np.ascontiguousarray(w.cell_type, dtype=np.uint8)).cuda()
    acc = ctypes.c_int64(-1)
    stream = torch.cuda.current_stream()
    rc = cpm.load().cpm_step_noalloc(ctypes.byref(cfg), lat.data_ptr(), V.data_ptr(), A.data_ptr(), ct.data_ptr(),
                                     0, 0, 7, ctypes.c_void_p(stream.cuda_stream), ctypes.byref(acc))
    assert rc == cpm.CPM_OK
    assert acc.value == st.replay_subpasses(7)
    torch.cuda.synchronize()
    assert np.array_equal(lat.cpu().numpy(), st.lattice)
    assert np.array_equal(V.cpu().numpy(), st.V) and np.array_equal(A.cpu().numpy(), st.A)
