"""Which calls on a large 3D lattice run in cubes: the way there and back are two launches of their own."""
import numpy as np
import pytest

from tests.test_gpu_cubes import _workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("act,perimeter", [(True, True), (False, False)])
def test_long_calls_run_in_cubes_and_short_ones_in_rows(act, perimeter):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    w = _workload((288, 272, 304), act, perimeter, 4)     # 95 MB, areas of 16^3
    n_sub = w.c ** 3 * w.P                                # sub-passes of an MCS
    k = (w.a // w.c) ** 3 // w.P                          # rounds of a sub-pass
    # attempts of half the sites or more, also over the end of an MCS
    calls = [(n_sub // 2 - 1, False), (n_sub // 2, True), (1, False), (n_sub, True), (n_sub // 8, False)]
    sim = cpm.Sim(w)
    clamped, at = act, 0                                  # the stamps' clamp, with sub-pass 0 of MCS 0 only
    for n, in_cubes in calls:
        before = sim.launches()
        sim.step_subpasses(n)
        assert sim.launches() - before == n * k + (2 if in_cubes else 0) + (1 if clamped else 0), (at, n)
        clamped, at = False, at + n
    lat = sim.read_lattice()
    sim.close()
    rows = cpm.Sim(w)
    for n in [n_sub // 8] * (at // (n_sub // 8)) + [1] * (at % (n_sub // 8)):
        rows.step_subpasses(n)
    assert np.array_equal(rows.read_lattice(), lat)
    rows.close()
