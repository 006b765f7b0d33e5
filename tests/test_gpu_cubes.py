"""Large 3D lattices run in cubes within a call of many rounds, in rows in calls
of few: the same lattice, Act values and tallies, bit for bit, whichever way an
MCS is cut into calls, from extents that are multiples of 8 but not of the
groups of cubes that are moved together."""
import numpy as np
import pytest

import cpm_workloads as cw

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


def _workload(shape, act, perimeter, seed):
    nx, ny, nz = shape
    rng = np.random.default_rng(seed)
    lat = np.zeros((nz, ny, nx), dtype=np.int32)
    cells = rng.permutation((nx // 8) * (ny // 8) * (nz // 8))[:60000]
    z, y, x = np.unravel_index(cells, (nz // 8, ny // 8, nx // 8))
    edge = 7
    for k in range(edge ** 3):
        o = np.unravel_index(k, (edge,) * 3)
        lat[(8 * z + o[0] - 3) % nz, (8 * y + o[1] - 3) % ny, (8 * x + o[2] - 3) % nx] = np.arange(1, len(cells) + 1)
    lat[rng.integers(0, nz, 4000), rng.integers(0, ny, 4000), rng.integers(0, nx, 4000)] = -1
    base = cw.random_small(11, dim=3, n=32, n_cells=8, edge=6, perimeter=perimeter, act=act, obstacles=0.02, a=16, c=2, P=64)
    actv = rng.integers(0, 5, lat.shape).astype(np.uint8) * (lat > 0) if act else None
    return base.replace(nx=nx, ny=ny, nz=nz, a=16, c=2, P=64, seed=seed, lattice=lat, act=actv,
                        cell_type=np.concatenate([[0], np.ones(len(cells))]).astype(np.uint8))


@pytest.mark.parametrize("shape,act,perimeter,track", [
    ((288, 320, 272), True, True, False),
    ((272, 288, 304), False, True, True),
    ((320, 272, 288), True, False, True),
])
def test_cubes_and_rows_give_the_same_lattice(cpm, shape, act, perimeter, track):
    w = _workload(shape, act, perimeter, 3)
    n_sub = w.c ** 3 * w.P                       # sub-passes of an MCS
    out = []
    for parts in ([n_sub], [n_sub // 8] * 8):    # at least half an MCS in a call runs in cubes
        sim = cpm.Sim(w)
        if track:
            sim.track_centroids(True)
        for n in parts:
            sim.step_subpasses(n)
        V, A = sim.read_tallies()
        got = [sim.read_lattice(), V, A, np.array([sim.stats()["accepts"]])]
        if act:
            got.append(sim.read_act())
        out.append([np.asarray(g) for g in got])
        sim.close()
    assert out[0][3][0] > 0
    for a, b in zip(*out):
        assert np.array_equal(a, b)
