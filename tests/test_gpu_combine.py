"""The combine where its rows are read in one or three vectors a pass: around the token counts of the rule, widths of one and of
several passes, dropped assignments, with and without gates' residual, in place."""
import pytest
import torch

from paper_2605_06665_b200 import binding as B

pytestmark = pytest.mark.gpu
SMS = 148


@pytest.mark.parametrize("T,d,k", [
    (1, 64, 5), (33, 768, 8), (8 * SMS, 768, 5), (8 * SMS + 1, 768, 8), (16 * SMS, 832, 8), (16 * SMS + 1, 832, 6), (9 * SMS, 2944, 7),
    (1500, 448, 8), (1500, 384, 8), (700, 768, 4), (1300, 1088, 3),
])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("residual", ["none", "other", "in place"])
def test_combine_by_vectors_a_pass(T, d, k, dtype, residual):
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    ctx = B.Context(B.make_config(d, 64, 16, k, 1, T, B.BF16 if dtype == "bf16" else B.FP32, 1e-6, 2.0))
    g = torch.Generator(device="cuda").manual_seed(T + d)
    n = 500                                             # rows in use
    Yp = torch.randn(n, d, device="cuda", generator=g).to(td)
    row_of = torch.randint(-1, n, (T, k), device="cuda", generator=g).to(torch.int32)
    gate = torch.rand(T, k, device="cuda", generator=g)
    x = torch.randn(T, d, device="cuda", generator=g).to(td)
    y = x.clone() if residual == "in place" else torch.full((T, d), float("nan"), device="cuda", dtype=td)
    ctx.combine(Yp, row_of, gate, T, {"none": None, "other": x, "in place": y}[residual], y)
    torch.cuda.synchronize()
    ctx.close()
    want = torch.zeros(T, d, device="cuda", dtype=torch.float64) if residual == "none" else x.double()
    size = want.abs()
    for j in range(k):
        term = torch.where(row_of[:, j:j + 1] >= 0, gate[:, j:j + 1].double() * Yp[row_of[:, j].clamp(min=0).long()].double(), 0.0)
        want, size = want + term, size + term.abs()
    # k + 1 terms added in fp32, then rounded to the type: bf16 has 8 significant bits, half a unit of the last one is up to
    # 2^-8 of the value
    bound = (k + 1) * 2.0 ** -24 * size + (2.0 ** -8 * 1.01 * want.abs() if dtype == "bf16" else 0.0)
    assert ((y.double() - want).abs() <= bound + 1e-30).all()
