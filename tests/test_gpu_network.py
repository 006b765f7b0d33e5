"""The fused forward, training and weight-update kernels of the emulator
network against the same layers computed one by one through cpm_mlp_gemm, at
the edges of what they take: one row, rows around a tile and a slab, every
width, padded and full inputs, one and many hidden layers, both output widths,
pre-activations beyond the range of the packed GELU.

Both sides multiply the same bf16 operands and sum each element over K in
ascending order with the same 16-wide products, so outputs and weight
gradients are compared for equal bits.  Only sums whose order is free have a
tolerance: bias gradients and losses, n terms in float32: n 2^-23 sum|x|.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# members, inputs, width, hidden layers, outputs, rows, weight scale
CASES = [
    (5, 7, 256, 4, 16, 1024, 0.1),
    (5, 7, 256, 4, 16, 1000, 0.1),
    (2, 7, 64, 2, 16, 1, 0.2),
    (3, 7, 128, 3, 16, 129, 0.1),
    (2, 17, 192, 1, 32, 127, 0.1),
    (2, 32, 256, 5, 32, 640, 0.1),
    (1, 1, 64, 4, 16, 33, 0.2),
    (2, 16, 128, 2, 32, 2048, 3.0),   # |z| beyond 13
    (1, 7, 256, 15, 16, 100, 0.1),
    (16, 7, 64, 2, 16, 1500, 0.2),    # more tiles than SMs
]


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import build as B
    B.build()
    from paper_2312_09317_gb300 import cpm
    return cpm.load()


def _gemm(lib, ta, tb, m, n, k, A, B, bias=None, f32=False, Z=None, epi=0):
    """One member's product: C and, for a GELU epilogue, its pre-activations."""
    C = torch.empty((m, n), dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    assert A.is_contiguous() and B.is_contiguous()
    p = lambda t: t.data_ptr() if t is not None else None  # noqa: E731
    rc = lib.cpm_mlp_gemm(ta, tb, m, n, k, 1, p(A), m if ta else k, 0, p(B), k if tb else n, 0, p(bias), 0, p(C),
                          int(f32), n, 0, p(Z), n, 0, epi, None)
    assert rc == 0
    return C


def _layers(flat, sizes):
    out, o = [], 0
    for i, n in zip(sizes[:-1], sizes[1:]):
        W = torch.from_numpy(flat[o:o + i * n].reshape(n, i)).cuda()
        b = torch.from_numpy(flat[o + i * n:o + i * n + n]).cuda()
        out.append((W.to(torch.bfloat16).contiguous(), b.contiguous()))
        o += i * n + n
    return out


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_fused_layers_against_single_ones(lib, case):
    from paper_2312_09317_gb300 import emulator as em
    E, n_in, width, n_hidden, n_out, rows, scale = case
    sizes = [n_in] + [width] * n_hidden + [n_out]
    P = sum(i * o + o for i, o in zip(sizes[:-1], sizes[1:]))
    rng = np.random.default_rng(rows + width)
    init = (rng.standard_normal((E, P)) * scale).astype(np.float32)
    n_total = rows + 50
    X = torch.from_numpy(rng.standard_normal((n_total, n_in)).astype(np.float32)).cuda()
    Y = torch.from_numpy(rng.standard_normal((n_total, n_out)).astype(np.float32)).cuda()
    order = torch.from_numpy(rng.integers(0, n_total, 3 * rows).astype(np.int32)).cuda()
    e = em.Ensemble(init, E, n_in, width, n_hidden, n_out, max_rows=rows)
    out = e.forward(X)  # (more rows than max_rows)
    g, loss = e.grads(X, Y, order=order, offset=rows, rows=rows)
    batch = order[rows:2 * rows].long()
    inv = torch.tensor(1.0 / np.float32(rows * n_out), dtype=torch.float32, device="cuda")
    for m in range(E):
        L = _layers(init[m], sizes)

        def forward(x):
            H, Zs = [x.to(torch.bfloat16).contiguous()], []
            for l, (W, b) in enumerate(L):
                last = l == n_hidden
                Z = None if last else torch.empty((x.shape[0], width), dtype=torch.float32, device="cuda")
                H.append(_gemm(lib, 0, 1, x.shape[0], sizes[l + 1], sizes[l], H[-1], W, b, last, Z, 0 if last else 1))
                Zs.append(Z)
            return H, Zs

        H, _ = forward(X)
        assert torch.equal(out[m], H[-1])
        H, Zs = forward(X[batch])
        d = H[-1] - Y[batch]
        terms = (d.double() ** 2).cpu().numpy()
        assert abs(float(loss[m]) - terms.mean()) <= rows * n_out * 2.0 ** -23 * terms.mean()
        dz = (2.0 * d * inv).to(torch.bfloat16)
        grads = []
        for l in range(n_hidden, -1, -1):
            grads.append((_gemm(lib, 1, 0, sizes[l + 1], sizes[l], rows, dz, H[l], f32=True), dz))
            if l:
                dz = _gemm(lib, 0, 0, rows, sizes[l], sizes[l + 1], dz, L[l][0], Z=Zs[l - 1], epi=2)
        o = 0
        for l, (dW, dz) in enumerate(reversed(grads)):
            n = dW.numel()
            assert torch.equal(g[m, o:o + n].view_as(dW), dW), (m, l)
            o += n
            z = dz.double()
            err = (g[m, o:o + sizes[l + 1]].double() - z.sum(0)).abs()
            assert bool((err <= rows * 2.0 ** -23 * z.abs().sum(0)).all()), (m, l)
            o += sizes[l + 1]
    e.close()


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_training_keeps_the_packed_weights_in_step(lib, case):
    """After a few steps the network works on exactly its new weights: a fresh
    one that is given them has the same outputs and gradients."""
    from paper_2312_09317_gb300 import emulator as em
    E, n_in, width, n_hidden, n_out, rows, scale = case
    sizes = [n_in] + [width] * n_hidden + [n_out]
    P = sum(i * o + o for i, o in zip(sizes[:-1], sizes[1:]))
    rng = np.random.default_rng(rows + width + 1)
    init = (rng.standard_normal((E, P)) * scale).astype(np.float32)
    X = torch.from_numpy(rng.standard_normal((rows, n_in)).astype(np.float32)).cuda()
    Y = torch.from_numpy(rng.standard_normal((rows, n_out)).astype(np.float32)).cuda()
    order = torch.from_numpy(rng.integers(0, rows, 3 * rows).astype(np.int32)).cuda()
    e = em.Ensemble(init, E, n_in, width, n_hidden, n_out, max_rows=rows)
    trace = e.train(X, Y, order, rows, 1e-3, trace=True)
    assert trace.shape == (3, E) and bool(torch.isfinite(trace).all())
    w = e.get_params()
    assert not np.array_equal(w, init)
    f = em.Ensemble(w, E, n_in, width, n_hidden, n_out, max_rows=rows)
    assert torch.equal(e.forward(X), f.forward(X))
    assert torch.equal(e.grads(X, Y)[0], f.grads(X, Y)[0])
    e.close()
    f.close()
