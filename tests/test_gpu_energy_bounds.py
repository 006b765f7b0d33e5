"""Energies at the bounds of the round kernels' 32-bit arithmetic: lambda_Act one below its bound and Max_act 1 beside
127, so that the Act term reaches 2,032 lambda_Act (just below 2^30), added to volume terms of both signs beyond the
2^30 at which a sum is clamped.  Bit for bit against the replay, which adds in 64 bits."""
import numpy as np
import pytest

import cpm_workloads as cw
import oracle

torch = pytest.importorskip("torch")


def workload(dim, n, seed):
    rng = np.random.default_rng(seed)
    w = cw.random_small(seed, dim=dim, n=n, n_cells=24, edge=4 if dim == 2 else 3, act=True, a=4, P=1, T=2900.0)
    ids = w.lattice
    ma = np.zeros_like(w.max_act)
    ma[1:3] = 1, 127
    la = np.zeros_like(w.lambda_act)
    la[1:3] = (1 << 19) - 1
    lv, vt = w.lambda_v.copy(), w.v_target.copy()
    lv[1:3] = 1 << 25
    vt[1:3] = (12, 11) if dim == 2 else (18, 17)
    # full activity but for one site in thirty
    act = np.where(ids > 0, ma[w.cell_type[np.maximum(ids, 0)]], 0) * (rng.random(ids.shape) > 0.03)
    return w.replace(max_act=ma, lambda_act=la, lambda_v=lv, v_target=vt, act=act.astype(np.uint8))


CASES = [(2, 32, 571), (2, 32, 578), (3, 16, 577)]


@pytest.mark.parametrize("dim,n,seed", CASES)
def test_the_workloads_reach_the_bounds(dim, n, seed):
    w = workload(dim, n, seed)
    st = oracle.State(w.replace(T=20.0))  # (no term depends on T)
    flat, offs = w.lattice.ravel(), oracle.neighbour_offsets(dim)
    dh, act = [], []
    for j in np.random.default_rng(seed).permutation(flat.size):
        j = int(j)
        x, y, z = j % w.nx, j // w.nx % w.ny, j // (w.nx * w.ny)
        for k, o in enumerate(offs):
            i = (x + o[0]) % w.nx + w.nx * ((y + o[1]) % w.ny + w.ny * ((z + (o[2] if dim == 3 else 0)) % w.nz))
            if flat[i] != flat[j]:
                d = st.delta_h(j, k)
                dh.append(16 * d["dh_int"])
                act.append(d["dh_act_q"])
    dh, act = np.array(dh), np.array(act)
    near = act > 0.999 * 2032 * ((1 << 19) - 1)
    assert near.any() and act.max() < 1 << 30 and act.min() > -(1 << 23)
    assert (dh[near] > 1 << 30).any() and (dh[near] < -(1 << 30)).any()
    assert (np.abs(dh + act) < 1 << 28).any()  # and sums that the term decides


@pytest.mark.gpu
@pytest.mark.parametrize("dim,n,seed", CASES)
def test_energies_at_the_bounds(dim, n, seed):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    w = workload(dim, n, seed)
    sim, ref = cpm.Sim(w), oracle.State(w)
    for step in range(1, 5):
        sim.step(step)
        ref.replay_run(step)
        V, A = sim.read_tallies()
        assert np.array_equal(sim.read_lattice(), ref.lattice)
        assert np.array_equal(V, ref.V) and np.array_equal(A, ref.A)
        assert np.array_equal(sim.read_act(), ref.act)
        assert sim.stats()["accepts"] == ref.accepts
    sim.close()
