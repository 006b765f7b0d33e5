"""Observations of a cell that reaches far along the axis that is walked: the squares of its sites' offsets from
its first site pass 32 bits when 16 of them are added, and then singly.  Bit-exact against the oracle."""
import numpy as np
import pytest

import cpm_workloads as cw
from oracle import observe as oobs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,length", [((64, 30016, 1), 29000), ((8, 8, 24000), 23000), ((4, 100000, 1), 99000),
                                          ((64, 16400, 1), 16399)])
def test_a_cell_along_a_long_axis(shape, length):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    nx, ny, nz = shape
    dim = 3 if nz > 1 else 2
    lat = np.zeros((nz, ny, nx), dtype=np.int32)
    if dim == 3:
        lat[:length, 1, 2] = 1
        lat[5:90, 4, 5] = 2
    else:
        lat[0, :length, 2] = 1
        lat[0, 5:90, 0] = 2
    base = cw.random_small(7, dim=dim, n=16, n_cells=4, edge=3, perimeter=True, a=4, c=2, P=4)
    w = base.replace(nx=nx, ny=ny, nz=nz, a=4, c=2, P=1, lattice=lat, act=None,
                     cell_type=np.array([0, 1, 1], dtype=np.uint8))
    b = cpm.Batch([w])
    cells = torch.empty((3, cpm.OBS_FIELDS), dtype=torch.int64, device="cuda")
    member = torch.empty((1, 2), dtype=torch.int64, device="cuda")
    b.observe(cells, member)
    torch.cuda.synchronize()
    assert np.array_equal(cells.cpu().numpy(), oobs.cell_rows(lat, w.n_cells, dim))
    assert int(member[0, 0]) == oobs.cell_medium_pairs(lat, dim)
    b.close()
