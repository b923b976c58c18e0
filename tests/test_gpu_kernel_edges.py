"""Small GPU tests at the sizes where a kernel or a branch of its dispatch can go wrong (edges of tiles,
remainders, unaligned inputs), each against a plain restatement or the aligned path."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,M,d", [(130, 5, 64), (130, 96, 192), (513, 5, 64), (513, 96, 192)])
@pytest.mark.parametrize("prepared", [False, True])
def test_router_terms_of_unaligned_fp32_weights(T, M, d, prepared):
    """Router weights that are not 16-byte aligned: same logits, bit for bit.  513 tokens read their bf16 terms, split by the
    scalar branch, 130 the weights themselves (the router for few tokens)."""
    import torch
    from paper_2605_06665_b200 import binding as B
    L = 2
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
        ctx.profile_enable(True)
        ctx.route(x, T, w[M * d:], 1.0, None, M, *o.values())
        assert ctx.profile_read()["route_logits"][1] == (1 if T > 464 and not prepared else 0)      # the split
        ctx.profile_enable(False)
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


# group sizes (k = 1, so rows = tokens) around the steps of the weights-on-M kernels: 16 and 32 tokens, 192 / 256 /
# 384 per unit, one and two MMAs, empty groups; the average decides the dispatch, so both layouts run
@pytest.mark.parametrize("sizes,d,f", [
    ([0, 1, 15, 16, 17, 31, 33, 191, 192, 193, 255, 256, 257, 383, 384, 385], 128, 1088),
    ([129, 512, 513, 0, 639, 640, 300], 192, 576),               # partial weight tiles
    ([768, 769, 1000, 1, 1152, 1153, 900], 1024, 64),            # gate/up beyond 450 rows, one k-block of K = 64
    ([200] * 40 + [0, 97, 1300], 64, 1216),
    ([110, 120, 130, 140], 256, 320),                            # both dgrads
    ([48, 1, 0, 33, 64, 65, 17], 128, 576),                      # both dgrads, few rows: stages of two k-blocks
    ([20, 1, 0, 33, 16, 5, 17], 192, 1216),                      # odd numbers of k-blocks in such stages
    ([384, 1, 0, 33, 16, 5, 17] * 3, 64, 1088),                  # one large unit among small ones
])
@pytest.mark.parametrize("with_rows", [True, False])
def test_expert_ffn_at_the_edges_of_its_units(sizes, d, f, with_rows):
    """Forward and both dgrads against a float32 restatement with the same bf16 roundings.  The kernels round
    G, U, A, Y, dGU and dX once each: |error| <= 2^-8 of the largest value plus the inputs' share, 1e-2."""
    import torch
    from paper_2605_06665_b200 import binding as B
    torch.backends.cuda.matmul.allow_tf32 = False
    M, T = len(sizes), sum(sizes)
    base, pool = 1, len(sizes) + 2
    ctx = B.Context(B.make_config(d, f, pool, 1, 1, T, B.BF16, 1e-6, 2.0))
    cap = ctx.row_capacity
    g = torch.Generator(device="cuda").manual_seed(5)
    bf = lambda *s, std=1.0: torch.empty(*s, device="cuda").normal_(0, std, generator=g).bfloat16()
    i32 = dict(dtype=torch.int32, device="cuda")
    x, dy = bf(T, d), bf(T, d)
    Wgu, Wd = bf(pool, 2 * f, d, std=0.05), bf(pool, d, f, std=0.05)
    idx = torch.repeat_interleave(torch.arange(M), torch.tensor(sizes))[torch.randperm(T)].to(torch.int32).cuda()[:, None]
    off, row_of, tok, te, rows = (torch.empty(s, **i32) for s in ((M + 1,), (T, 1), (cap,), (cap // 128,), (M,)))
    nan = lambda *s: torch.full(s, float("nan"), dtype=torch.bfloat16, device="cuda")
    Xp, GU, A, Yp, dYp, dGU, dx = nan(cap, d), nan(cap, 2 * f), nan(cap, f), nan(cap, d), nan(cap, d), nan(cap, 2 * f), nan(T, d)
    gate, dgate = torch.rand(T, 1, device="cuda", generator=g) + 0.5, torch.empty(T, 1, device="cuda")
    ctx.dispatch(x, T, idx.contiguous(), M, off, row_of, tok, te, Xp, rows)
    assert rows.tolist() == sizes
    r = rows if with_rows else None
    ctx.expert_fwd(Xp, off, te, Wgu, Wd, base, M, GU, A, Yp, r)
    ctx.expert_bwd(dy, T, row_of, gate, tok, off, te, Xp, GU, A, Yp, Wgu, Wd, base, M, None, dYp, dGU, dx, dgate, None,
                   None, B.BWD_SKIP_WGRAD, r)
    torch.cuda.synchronize()
    ctx.check_status()
    ctx.close()
    off = off.tolist()
    used = off[-1]
    pad = tok[:used] < 0
    for t in (Xp, GU, A, Yp):
        assert not t[:used][pad].any()                            # zeros (and no NaN) on pad rows
    if with_rows:                                                 # of dYp, dGU those up to the next multiple of 16 rows
        for e, n in enumerate(sizes):
            pad[off[e] + (n + 15) // 16 * 16:off[e + 1]] = False
    for t in (dYp, dGU):
        assert not t[:used][pad].any()

    def close(got, want):
        assert (got.float() - want.float()).abs().max() <= 1e-2 * want.float().abs().max()

    for e, n in enumerate(sizes):
        if n == 0:
            continue
        s = slice(off[e], off[e] + n)
        X, Wg, Wu, W2 = (t.float() for t in (Xp[s], Wgu[base + e, :f], Wgu[base + e, f:], Wd[base + e]))
        G, U = X @ Wg.T, X @ Wu.T
        close(GU[s, :f], G)
        close(GU[s, f:], U)
        close(A[s], torch.nn.functional.silu(G) * U)
        close(Yp[s], A[s].float() @ W2.T)
        dA = dYp[s].float() @ W2
        G, U = GU[s, :f].float(), GU[s, f:].float()
        sig = torch.sigmoid(G)
        close(dGU[s, :f], dA * U * sig * (1 + G * (1 - sig)))
        close(dGU[s, f:], dA * G * sig)
        close(dx[tok[s].long()], dGU[s].float() @ Wgu[base + e].float())


@pytest.mark.parametrize("overwrite", [True, False])
@pytest.mark.parametrize("sizes", [
    [[0, 0, 0, 0], [0, 0, 0, 0]],
    [[1, 15, 16, 17], [63, 64, 65, 0], [0, 127, 128, 129], [33, 0, 48, 1000]],
    [[5, 0, 7, 200]],
    [[1, 31, 32, 33], [0, 47, 48, 10]],                # 26 rows per expert: k-blocks of 32
    [[33, 47, 48, 17], [49, 1, 95, 0], [0, 0, 0, 7]],  # 36: k-blocks of 48
])
def test_weight_gradient_leaves_the_padding_out(sizes, overwrite):
    """With the group sizes the contraction stops at the last 16 rows that hold a token, whatever the rest of the padding
    holds; what is left out of the padded contraction are zeros, so the sums are equal, bit for bit."""
    import torch
    from paper_2605_06665_b200 import binding as B
    L, M, d, f = len(sizes), 4, 192, 320
    T = max(sum(s) for s in sizes)
    ctx = B.Context(B.make_config(d, f, M, 1, L, max(T, 1), B.BF16, 1e-6, 2.0))
    cap = ctx.row_capacity
    g = torch.Generator(device="cuda").manual_seed(2)
    off = np.zeros((L, M + 1), dtype=np.int32)
    for l, s in enumerate(sizes):
        off[l, 1:] = np.cumsum([(n + 127) // 128 * 128 for n in s])
    ops = [torch.zeros(L, cap, w, dtype=torch.bfloat16, device="cuda") for w in (d, f, d, 2 * f)]
    for l, s in enumerate(sizes):
        for e, n in enumerate(s):
            for t in ops:
                t[l, off[l, e]:off[l, e] + n].normal_(generator=g)
    rows = torch.tensor(sizes, dtype=torch.int32, device="cuda")
    offs = torch.from_numpy(off).cuda()
    got = []
    for r in (None, rows):
        if r is not None:
            for l, s in enumerate(sizes):
                for e, n in enumerate(s):
                    for t in ops:
                        t[l, off[l, e] + (n + 15) // 16 * 16:off[l, e + 1]] = float("nan")
        dgu, dd = torch.full((M, 2 * f, d), 3.0, device="cuda"), torch.full((M, d, f), -2.0, device="cuda")
        ctx.pool_wgrad(L, cap, offs, *ops, 0, M, dgu, dd, B.WGRAD_OVERWRITE if overwrite else 0, r)
        torch.cuda.synchronize()
        got.append((dgu, dd))
    ctx.check_status()
    ctx.close()
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    Xp, A, dYp, dGU = (t.float() for t in ops)
    for e in range(M):
        want = torch.zeros(2 * f, d, device="cuda") if overwrite else torch.full((2 * f, d), 3.0, device="cuda")
        down = torch.zeros(d, f, device="cuda") if overwrite else torch.full((d, f), -2.0, device="cuda")
        for l in range(L):
            s = slice(off[l, e], off[l, e] + sizes[l][e])
            want += dGU[l, s].T @ Xp[l, s]
            down += dYp[l, s].T @ A[l, s]
        # exact products, fp32 sums of at most some 1200 terms: 1e-5 of the largest value
        assert (got[1][0][e] - want).abs().max() <= 1e-5 * max(want.abs().max().item(), 1.0)
        assert (got[1][1][e] - down).abs().max() <= 1e-5 * max(down.abs().max().item(), 1.0)


@pytest.mark.parametrize("sizes,d,f", [
    ([0, 1, 15, 16, 17, 63, 64, 65, 127, 128, 129], 64, 64),      # narrow tiles, two groups of threads per tile
    ([500, 0, 700, 1, 2000, 64], 256, 512),                       # wide tiles
])
@pytest.mark.parametrize("shift", [0, 1])                         # 1: pointers that are not 16-byte aligned
def test_fp32_expert_ffn_at_the_edges_of_its_tiles(sizes, d, f, shift):
    """fp32 mode against float64.  Sums of at most 2000 products: |error| <= 2000 * 2^-24 of the terms' magnitudes,
    which random signs keep far below 1e-5 of the largest value."""
    import torch
    from paper_2605_06665_b200 import binding as B
    M, T = len(sizes), sum(sizes)
    ctx = B.Context(B.make_config(d, f, M, 1, 1, T, B.FP32, 1e-6, 2.0))
    cap = ctx.row_capacity
    g = torch.Generator(device="cuda").manual_seed(5)

    def new(*s, std=None):
        n = int(np.prod(s))
        t = torch.full((n + 4,), float("nan"), device="cuda")[shift:shift + n].view(s)
        return t if std is None else t.normal_(0, std, generator=g)

    i32 = dict(dtype=torch.int32, device="cuda")
    x, dy = torch.randn(T, d, device="cuda", generator=g), torch.randn(T, d, device="cuda", generator=g)
    Wgu, Wd = new(M, 2 * f, d, std=0.05), new(M, d, f, std=0.05)
    idx = torch.repeat_interleave(torch.arange(M), torch.tensor(sizes))[torch.randperm(T)].to(torch.int32).cuda()[:, None].contiguous()
    off, row_of, tok, te, rows = (torch.empty(s, **i32) for s in ((M + 1,), (T, 1), (cap,), (cap // 128,), (M,)))
    rowbuf = lambda w: torch.full((cap, w), float("nan"), device="cuda")
    Xp, Yp, dYp, dx = rowbuf(d), rowbuf(d), rowbuf(d), torch.empty(T, d, device="cuda")
    GU, A, dGU = new(cap, 2 * f), new(cap, f), new(cap, 2 * f)
    dWgu, dWd = new(M, 2 * f, d), new(M, d, f)
    gate, dgate = torch.rand(T, 1, device="cuda", generator=g) + 0.5, torch.empty(T, 1, device="cuda")
    ctx.dispatch(x, T, idx, M, off, row_of, tok, te, Xp, rows)
    ctx.expert_fwd(Xp, off, te, Wgu, Wd, 0, M, GU, A, Yp, rows)
    ctx.expert_bwd(dy, T, row_of, gate, tok, off, te, Xp, GU, A, Yp, Wgu, Wd, 0, M, None, dYp, dGU, dx, dgate, dWgu, dWd,
                   B.WGRAD_OVERWRITE, rows)
    torch.cuda.synchronize()
    ctx.check_status()
    ctx.close()
    used = int(off[-1])
    pad = tok[:used] < 0
    for t in (GU, A, Yp, dGU):
        assert not t[:used][pad].any()

    def close(got, want):
        assert (got.double() - want).abs().max() <= 1e-5 * max(want.abs().max().item(), 1e-3)

    for e, n in enumerate(sizes):
        s = slice(int(off[e]), int(off[e]) + n)
        X, Wg, Wu, W2, dY = (t.double() for t in (Xp[s], Wgu[e, :f], Wgu[e, f:], Wd[e], dYp[s]))
        if n:
            G, U = X @ Wg.T, X @ Wu.T
            close(GU[s], torch.cat([G, U], 1))
            close(A[s], torch.nn.functional.silu(G) * U)
            close(Yp[s], A[s].double() @ W2.T)
            G, U, dA = GU[s, :f].double(), GU[s, f:].double(), dY @ W2
            sig = torch.sigmoid(G)
            close(dGU[s], torch.cat([dA * U * sig * (1 + G * (1 - sig)), dA * G * sig], 1))
            close(dx[tok[s].long()], dGU[s].double() @ Wgu[e].double())
        close(dWd[e], dY.T @ A[s].double())
        close(dWgu[e], dGU[s].double().T @ X)


@pytest.mark.parametrize("T,M,d", [(1, 1, 64), (33, 13, 128), (512, 16, 256), (1100, 33, 64), (2100, 36, 192)])
@pytest.mark.parametrize("shift", [0, 1])
def test_fp32_router_products_at_the_edges_of_their_tiles(T, M, d, shift):
    """Logits, dx and dW_r of the fp32 router: M with and without 16-byte rows of dz, tokens beyond one run of 1024,
    router weights that are not 16-byte aligned; against the oracle in float64 (1e-5, as in the parity tests)."""
    import torch
    from oracle import unipool_oracle as O
    from paper_2605_06665_b200 import binding as B
    k, c, eps = 1, 2.0, 1e-6
    ctx = B.Context(B.make_config(d, 64, M, k, 1, T, B.FP32, eps, c))
    g = torch.Generator(device="cuda").manual_seed(T)
    W = torch.empty(M * d + 4, device="cuda")[shift:shift + M * d].view(M, d).normal_(0, 0.02, generator=g)
    x, dgate = torch.randn(T, d, device="cuda", generator=g), torch.randn(T, k, device="cuda", generator=g)
    idx = torch.empty(T, k, dtype=torch.int32, device="cuda")
    gate, counts = torch.empty(T, k, device="cuda"), torch.empty(M, dtype=torch.int32, device="cuda")
    S, n, z = torch.empty(M, device="cuda"), torch.empty(T, device="cuda"), torch.empty(T, M, device="cuda")
    coef = torch.rand(M, device="cuda", generator=g)
    dx, dW, dsig = torch.ones(T, d, device="cuda"), torch.full((M, d), 2.0, device="cuda"), torch.zeros(1, device="cuda")
    ctx.route(x, T, W, 1.0, None, M, idx, gate, counts, S, n, z)
    ctx.route_bwd(x, T, W, 1.0, M, n, z, idx, dgate, coef, dx, dW, dsig)
    torch.cuda.synchronize()
    ctx.check_status()
    ctx.close()
    f8 = lambda t: t.double().cpu().numpy()
    ref = O.route(f8(x), f8(W), 1.0, c, eps, k, None, forced_idx=idx.cpu().numpy())
    rb = O.route_backward(f8(x), f8(W), 1.0, c, eps, ref["z"], ref["n"], idx.cpu().numpy(), f8(dgate), f8(coef))
    for got, want in ((z, ref["z"]), (dx - 1, rb["dx"]), (dW - 2, rb["dW_r"])):
        scale = max(np.abs(want).max(), 1.0 if want is not ref["z"] else 0.0)       # dx and dW were added to 1 and 2
        assert np.abs(f8(got) - want).max() <= 1e-5 * scale


@pytest.mark.parametrize("kw,L,T", [
    (dict(M=48, k=1), 5, 40),                       # runs of two, two and one layer
    (dict(M=32, k=2), 4, 70),
    (dict(M=64, k=2, groups=2), 6, 50),             # two sharing groups of three layers, runs of two and one
])
@pytest.mark.parametrize("accumulate", [False, True])
def test_recomputed_layers_contract_in_runs(kw, L, T, accumulate):
    """With recompute the weight gradients of a run of layers are contracted together: same sums as layer by layer up
    to the order of fp32 additions (1e-5, as for the one-pass contraction)."""
    import torch
    from paper_2605_06665_b200 import synth
    from paper_2605_06665_b200.stack import UniPoolStack
    from parity_utils import rel_max, to_np
    cfg = dict(L=L, d=256, f=384, T=T, dtype="bf16", private=0, zipf_beta=0.0, **kw)
    inputs = synth.make_inputs(cfg, seed=4, T=T)
    x0, up = (torch.from_numpy(inputs[n]).cuda().bfloat16() for n in ("x0", "upstream"))
    out = []
    for recompute in (False, True):
        st = UniPoolStack(L, 256, 384, kw["M"], kw["k"], T, "bf16", 0, c=2.5, recompute=recompute, groups=kw.get("groups"))
        st.load(inputs["pool"], inputs["routers"])
        if recompute:
            assert 1 < st.nw <= st.Lg and st.GU.shape[0] == st.Yp.shape[0] == 1
        if accumulate:
            st.zero_grad()
        else:
            st.dW_gu.fill_(11.0); st.dW_down.fill_(-2.0)
        dx = st.step(x0, up, accumulate=accumulate).clone()
        torch.cuda.synchronize()
        st.ctx.check_status()
        out.append((dx, st.dW_gu.clone(), st.dW_down.clone()))
        st.close()
    assert torch.equal(out[0][0], out[1][0]) and out[0][1].abs().max() > 0
    assert rel_max(to_np(out[1][1]), to_np(out[0][1])) < 1e-5 and rel_max(to_np(out[1][2]), to_np(out[0][2])) < 1e-5


@pytest.mark.parametrize("T,M,d,k", [
    (1, 8, 64, 8), (257, 10, 64, 3), (130, 256, 128, 8), (300, 257, 128, 5), (520, 512, 64, 8), (300, 384, 832, 8), (33, 96, 768, 2),
    (465, 8, 64, 8), (513, 10, 64, 3), (700, 256, 128, 8), (600, 257, 128, 5), (640, 384, 832, 8), (465, 96, 768, 2), (1025, 9, 192, 1),
])
@pytest.mark.parametrize("bits", ["bf16", "fp32"])                # one or three bf16 terms of the router weights
@pytest.mark.parametrize("mode", ["norm", "softmax"])
def test_bf16_router_at_the_edges_of_its_stages(T, M, d, k, bits, mode):
    """Selection with many candidates per lane, one and two MMAs per k-block, one or three weight terms, fewer
    k-blocks than stages; against the oracle in float64 as in the parity tests.  (From 465 tokens on the tensor cores, below
    on clusters of CUDA-core blocks.)"""
    import torch
    from oracle import unipool_oracle as O
    from paper_2605_06665_b200 import binding as B
    from parity_utils import check_routing, rel_max, to_np
    eps, c = 1e-6, 2.0
    ctx = B.Context(B.make_config(d, 64, M, k, 1, T, B.BF16, eps, c, B.ROUTER_SOFTMAX if mode == "softmax" else B.ROUTER_NORM))
    g = torch.Generator(device="cuda").manual_seed(T)
    W = torch.empty(M, d, device="cuda").normal_(0, 0.02, generator=g)
    if bits == "bf16":
        W = W.bfloat16().float()
    x = torch.randn(T, d, device="cuda", generator=g).bfloat16()
    idx, gate = torch.empty(T, k, dtype=torch.int32, device="cuda"), torch.empty(T, k, device="cuda")
    counts, S = torch.empty(M, dtype=torch.int32, device="cuda"), torch.empty(M, device="cuda")
    n, z = torch.empty(T, device="cuda"), torch.empty(T, M, device="cuda")
    ctx.profile_enable(True)
    ctx.route(x, T, W, 1.0, None, M, idx, gate, counts, S, n, z)
    assert ctx.profile_read()["route_logits"][1] == (1 if T > 464 else 0)               # the tensor-core router splits W
    ctx.check_status()
    ctx.close()
    f8 = lambda t: t.double().cpu().numpy()
    ref = O.route(f8(x), f8(W), 1.0, c, eps, k, None, mode=mode)
    check_routing(to_np(idx), ref["z"], ref["idx"], k, mode)
    ref = O.route(f8(x), f8(W), 1.0, c, eps, k, None, forced_idx=to_np(idx), mode=mode)
    assert rel_max(to_np(z), ref["z"]) < 1e-5 and rel_max(to_np(gate), ref["g"]) < 1e-5
    assert (to_np(counts) == ref["counts"]).all() and rel_max(to_np(S), ref["S"]) < 1e-5
