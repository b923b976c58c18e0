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


@pytest.mark.parametrize("T,k,M", [
    (1, 1, 1), (1, 8, 8), (33, 2, 96), (512, 8, 9), (513, 8, 9),        # 512 * 8 = 4096: every block counts all indices
    (2048, 2, 5), (2049, 2, 512), (2368, 3, 40), (9472, 1, 7), (40000, 2, 33),   # chunks of 16 .. 256 tokens
])
@pytest.mark.parametrize("static", [False, True])
def test_dispatch_maps_at_the_edges_of_its_chunking(T, k, M, static):
    import torch
    from oracle import unipool_oracle as O
    from paper_2605_06665_b200 import binding as B
    d = 64
    ctx = B.Context(B.make_config(d, 64, M, k, 1, T, B.BF16, 1e-6, 2.0))
    cap = ctx.row_capacity
    rng = np.random.default_rng(T + k)
    p = rng.random(M) ** 3 + 1e-3
    idx = np.argsort(-np.log(p / rng.exponential(size=(T, M))), axis=1)[:, :k].astype(np.int32)      # distinct, skewed
    x = torch.empty(T, d, device="cuda").normal_(generator=torch.Generator(device="cuda").manual_seed(1)).bfloat16()
    i32 = dict(dtype=torch.int32, device="cuda")
    off, row_of, tok, te = (torch.full(s, -7, **i32) for s in ((M + 1,), (T, k), (cap,), (cap // 128,)))
    Xp = torch.full((cap, d), 3.0, dtype=torch.bfloat16, device="cuda")
    args = (off, row_of, tok, te, Xp)
    gi = torch.from_numpy(np.ascontiguousarray(idx)).cuda()
    if static:
        B.dispatch_static(x, T, d, B.BF16, k, gi, M, cap, *args)
    else:
        ctx.dispatch(x, T, gi, M, *args)
    torch.cuda.synchronize()
    ctx.check_status()
    ctx.close()
    r_off, r_row, r_tok = O.dispatch_map(idx, M, 128)
    used = int(r_off[-1])
    assert (off.cpu().numpy() == r_off).all() and (row_of.cpu().numpy() == r_row).all()
    assert (tok[:used].cpu().numpy() == r_tok).all() and (tok[used:] == -1).all()
    t = torch.from_numpy(r_tok.astype(np.int64)).cuda()
    want = torch.where((t >= 0)[:, None], x[t.clamp(min=0)], torch.zeros((), dtype=x.dtype, device="cuda"))
    assert torch.equal(Xp[:used], want)
    exp = np.full(cap // 128, -1)
    for e in range(M):
        exp[r_off[e] // 128:r_off[e + 1] // 128] = e
    assert (te.cpu().numpy() == exp).all()
