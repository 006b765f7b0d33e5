"""Observations where the walks of a CTA meet more cells than its shared sums
hold, where a lattice is too long for 32-bit sums, where runs end at every site
and where the last walk of an axis is short: bit-exact against the oracle."""
import numpy as np
import pytest

import cpm_workloads as cw
from oracle import observe as oobs

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


# extents, cells, edge of the blocks of one cell, Act
SHAPES = [
    ((64, 48, 20), 3000, 1, False),    # some 3,000 cells in a CTA's 4,096 sites
    ((64, 48, 20), 3000, 1, True),
    ((8, 8, 1032), 40, 4, False),      # 64-bit sums
    ((40, 24, 36), 150, 4, True),      # about the number that the shared sums hold
    ((128, 64, 24), 60, 8, False),
    ((8, 1032, 1), 300, 1, False),     # 2D
    ((52, 40, 1), 30, 4, True),
]


@pytest.mark.parametrize("shape,n_cells,edge,act", SHAPES)
def test_observations_at_the_walks_edges(cpm, shape, n_cells, edge, act):
    nx, ny, nz = shape
    dim = 3 if nz > 1 else 2
    rng = np.random.default_rng(nx + nz + n_cells)
    blocks = rng.integers(0, n_cells + 1, [-(-n // edge) for n in (nz, ny, nx)])
    lat = blocks.repeat(edge, 0).repeat(edge, 1).repeat(edge, 2)[:nz, :ny, :nx].astype(np.int32)
    lat.ravel()[rng.choice(lat.size, n_cells, replace=False)] = np.arange(1, n_cells + 1)  # every cell is there
    base = cw.random_small(7, dim=dim, n=16, n_cells=4, edge=3, perimeter=True, act=act, a=4, c=2, P=4)
    w = base.replace(nx=nx, ny=ny, nz=nz, a=4, c=2, P=1, lattice=lat, act=None,
                     cell_type=np.concatenate([[0], np.ones(n_cells)]).astype(np.uint8))
    b = cpm.Batch([w])
    rows = int(b.observation_rows()[-1])
    cells = torch.empty((rows, cpm.OBS_FIELDS), dtype=torch.int64, device="cuda")
    member = torch.empty((1, 2), dtype=torch.int64, device="cuda")
    b.observe(cells, member)
    torch.cuda.synchronize()
    assert np.array_equal(cells.cpu().numpy(), oobs.cell_rows(lat, w.n_cells, dim))
    assert int(member[0, 0]) == oobs.cell_medium_pairs(lat, dim)
    b.close()
