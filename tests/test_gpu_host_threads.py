"""Two host threads, each with handles and a stream of its own, whose calls need different amounts of shared memory
of the same kernels: every call succeeds and gives the bits that it gives alone."""
import threading

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


def _in_two_threads(calls, rounds):
    """Each call in a thread of its own, `rounds` times: the results of every tenth of them are those of the call alone."""
    def read(t):
        torch.cuda.synchronize()  # the calls' streams are not the one that copies
        return t.cpu().numpy()

    alone = [read(c()) for c in calls]
    faults, start = [], threading.Barrier(len(calls))

    def work(call, expected):
        try:
            start.wait()
            for k in range(rounds):
                got = call()
                if k % (rounds // 10) == 0:
                    assert np.array_equal(read(got), expected, equal_nan=True)
        except BaseException as e:  # noqa: BLE001 (handed to the test's thread)
            faults.append(e)

    threads = [threading.Thread(target=work, args=a) for a in zip(calls, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not faults, faults[0]


def test_summaries_of_few_and_many_snapshots(cpm):
    def call(n_snap):
        stream = torch.cuda.Stream()
        batch = cpm.Batch([cw.point_cells_2d(seed=k, n=16, n_cells=4, a=4) for k in range(2)], stream=stream)
        rows = int(batch.observation_rows()[-1])
        with torch.cuda.stream(stream):
            cells = torch.empty((n_snap, rows, cpm.OBS_FIELDS), dtype=torch.int64, device="cuda")
            member = torch.empty((n_snap, 2, 2), dtype=torch.int64, device="cuda")
            out = torch.empty((2, 16), dtype=torch.float64, device="cuda")
            for s in range(n_snap):
                batch.observe(cells[s], member[s])
        stream.synchronize()

        def run():
            with torch.cuda.stream(stream):
                batch.summarize(cells, member, 1, out)
                return out
        return run
    _in_two_threads([call(3), call(900)], 20000)


@pytest.mark.parametrize("what", ["forward", "grads"])
def test_networks_of_different_shapes(cpm, what):
    from paper_2312_09317_gb300 import emulator as em

    def call(E, width, n_hidden, rows):
        sizes = [7] + [width] * n_hidden + [16]
        stream = torch.cuda.Stream()
        net = em.Ensemble(cw.mlp_init(3, E, sizes), E, 7, width, n_hidden, 16, max_rows=rows, stream=stream)
        rng = np.random.default_rng(rows)
        with torch.cuda.stream(stream):
            X = torch.from_numpy(rng.uniform(0, 1, (rows, 7)).astype(np.float32)).cuda()
            Y = torch.from_numpy(rng.normal(0, 1, (rows, 16)).astype(np.float32)).cuda()
        stream.synchronize()

        def run():
            with torch.cuda.stream(stream):
                return net.forward(X) if what == "forward" else net.grads(X, Y)[0]
        return run
    _in_two_threads([call(1, 64, 1, 16), call(2, 256, 15, 300)], 5000)
