"""Small GPU tests at the sizes where a kernel or a branch of its dispatch can go wrong (edges of tiles,
remainders, unaligned inputs), each against a plain restatement or the aligned path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,d", [(5, 64), (96, 192)])
@pytest.mark.parametrize("prepared", [False, True])
def test_router_terms_of_unaligned_fp32_weights(M, d, prepared):
    """Router weights that are not 16-byte aligned are split by the scalar branch: same logits, bit for bit."""
    import torch
    from paper_2605_06665_b200 import binding as B
    T, L = 130, 2
    ctx = B.Context(B.make_config(d, 64, M, 1, L, T, B.BF16, 1e-6, 2.0))
    g = torch.Generator(device="cuda").manual_seed(3)
    W = torch.empty(L * M * d, device="cuda").normal_(0, 0.02, generator=g)
    x = torch.empty(T, d, device="cuda").normal_(generator=g).bfloat16()
    shifted = torch.empty(L * M * d + 1, device="cuda")[1:].copy_(W)
    out = []
    for w in (W, shifted):
        if prepared:
            ctx.router_prepare(w, L, M)
        o = dict(idx=torch.empty(T, 1, dtype=torch.int32, device="cuda"), gate=torch.empty(T, 1, device="cuda"),
                 counts=torch.empty(M, dtype=torch.int32, device="cuda"), score_sum=torch.empty(M, device="cuda"),
                 znorm=torch.empty(T, device="cuda"), z=torch.empty(T, M, device="cuda"))
        ctx.route(x, T, w[M * d:], 1.0, None, M, *o.values())
        torch.cuda.synchronize()
        out.append(o)
    ctx.check_status()
    ctx.close()
    for n in out[0]:
        assert torch.equal(out[0][n], out[1][n]), n
    ref = x.double() @ W[M * d:].reshape(M, d).double().T
    # fp32 sums of d exact products: |error| <= d * 2^-24 * sum |x w|, far below 1e-5 of the largest logit
    assert (out[0]["z"].double() - ref).abs().max() <= 1e-5 * ref.abs().max()
