"""Forward products whose K is 8 above a multiple of 16, the depth of a tensor-core step: what lies behind A's rows
(the columns up to its leading dimension, the memory behind its last row) takes no part in them, NaN as it may be.
A lies inside a larger buffer, so that every column that could be read belongs to the test."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [8, 16, 24, 40, 248])
@pytest.mark.parametrize("pad", [0, 8, 16])
@pytest.mark.parametrize("m", [1, 128, 300])
def test_columns_behind_k_take_no_part(m, pad, k):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2312_09317_gb300 import cpm
    lib = cpm.load()
    n, ld = 32, k + pad
    gen = torch.Generator(device="cuda").manual_seed(m + k)
    A = torch.randn((m, k), generator=gen, device="cuda").to(torch.bfloat16)
    B = torch.randn((n, k), generator=gen, device="cuda").to(torch.bfloat16)
    out = []
    for fill in (0.0, float("nan")):
        buf = torch.full((m * ld + 64,), fill, dtype=torch.bfloat16, device="cuda")
        buf[:m * ld].view(m, ld)[:, :k] = A
        C = torch.empty((m, n), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        assert lib.cpm_mlp_gemm(0, 1, m, n, k, 1, buf.data_ptr(), ld, 0, B.data_ptr(), k, 0, None, 0, C.data_ptr(), 1, n, 0,
                                None, n, 0, 0, None) == 0
        torch.cuda.synchronize()
        out.append(C)
    assert torch.equal(out[0], out[1])
    # k products of bf16 operands, exact in float32, and k - 1 roundings of their sum
    ref = A.double() @ B.double().T
    assert bool(((out[0].double() - ref).abs() <= k * 2.0 ** -23 * (A.double().abs() @ B.double().abs().T)).all())
