"""Both routers of the bf16 mode on values out of the ordinary: score sums beyond what their accumulators hold, infinite and NaN
logits, masked experts, ties."""
import numpy as np
import pytest
import torch

from oracle import unipool_oracle as O
from parity_utils import f64, to_np
from paper_2605_06665_b200 import binding as B

pytestmark = pytest.mark.gpu


def route(ctx, x, W, bias, k, sigma=1.0, few=None):
    """The call's outputs; few: which of the routers has to take it (only the other one splits the weights it is given)."""
    T, M = x.shape[0], W.shape[0]
    nan = lambda *s: torch.full(s, float("nan"), device="cuda")
    out = dict(idx=torch.full((T, k), -7, dtype=torch.int32, device="cuda"), gate=nan(T, k),
               counts=torch.full((M,), -7, dtype=torch.int32, device="cuda"), S=nan(M), n=nan(T), z=nan(T, M))
    ctx.profile_enable(True)
    ctx.route(x, T, W, sigma, bias, M, *(out[n] for n in ("idx", "gate", "counts", "S", "n", "z")))
    splits = ctx.profile_read()["route_logits"][1]
    ctx.profile_enable(False)
    assert few is None or splits == (0 if few else 1)
    return {n: to_np(t) for n, t in out.items()}


@pytest.mark.parametrize("T,sigma,fits", [(1, 2e10, True), (2, 2e10, False), (6, 5e9, True), (7, 5e9, False), (12, 2e10, False), (400, 5e9, False),
                                          (1, 4e10, False), (600, 2e8, False), (600, 4e7, True)])
def test_score_sums_at_the_range_of_their_accumulators(T, sigma, fits):
    """Sums are kept in multiples of 2^-28 in 64 bits: below 2^35 they are right, beyond it they are NaN, never a wrapped
    number; the next call finds clean accumulators."""
    ctx = B.Context(B.make_config(64, 64, 8, 1, 1, 600, B.BF16, 1e-6, 1.0, B.ROUTER_NORM))
    x, W = torch.zeros(T, 64, device="cuda", dtype=torch.bfloat16), torch.zeros(8, 64, device="cuda")
    x[:, 0] = W[3, 0] = 1.0
    out = route(ctx, x, W, None, 1, sigma, few=T <= 464)
    assert np.isnan(out["S"]).all() if not fits else abs(out["S"][3] / (T * sigma) - 1) < 1e-5 and out["S"][[0, 7]].tolist() == [0, 0]
    out = route(ctx, x, W, None, 1)
    assert abs(out["S"][3] / T - 1) < 1e-5 and out["counts"].tolist() == [0, 0, 0, T, 0, 0, 0, 0]
    ctx.close()


def special_bias(kind, M):
    b = np.zeros(M, np.float32)
    if kind == "negative": b[np.arange(M) != M // 2] = -600.0       # one logit above zero at most
    if kind == "infinite": b[3], b[M - 2], b[M // 2] = np.inf, -np.inf, -np.inf
    if kind == "nan": b[5] = np.nan
    if kind == "masked": b[:M - 9] = -np.inf                          # all experts of the first chunks of 32
    return b


@pytest.mark.parametrize("kind", ["ties", "negative", "infinite", "nan", "masked"])
@pytest.mark.parametrize("M,k", [(75, 2), (75, 8), (384, 2), (384, 8), (10, 2)])
@pytest.mark.parametrize("mode", ["norm", "softmax"])
def test_both_routers_agree_on_special_logits(mode, M, k, kind):
    """Logits that are whole numbers, the same in both kernels to the bit: selection is equal, everything else up to the rounding of
    sums (fp32, M terms of one sign: M / 2 ulp at most; score sums to multiples of 2^-28 in each of some 500 blocks).  Some tokens hold a NaN, an infinity, or nothing but zeros."""
    rng = np.random.default_rng(M + k)
    T, d = 500, 64
    ctx = B.Context(B.make_config(d, 64, M, k, 1, T, B.BF16, 1e-6, 1.0, B.ROUTER_SOFTMAX if mode == "softmax" else B.ROUTER_NORM))
    x = torch.from_numpy(rng.integers(0, 2, (T, d)).astype(np.float32)).cuda().bfloat16()
    W = torch.from_numpy(rng.integers(-1, 2, (M, d)).astype(np.float32)).cuda()
    x[7] = 0.0
    if kind != "masked":
        x[11, 2] = float("nan")
        x[13, 1] = float("inf")
    b = special_bias(kind, M)
    bias = torch.from_numpy(b).cuda()
    whole = route(ctx, x, W, bias, k, few=False)
    parts = [route(ctx, x[:40].contiguous(), W, bias, k, few=True), route(ctx, x[40:].contiguous(), W, bias, k, few=True)]
    few = {n: sum(p[n] for p in parts) if n in ("counts", "S") else np.concatenate([p[n] for p in parts]) for n in whole}
    tol = M * 2.0 ** -24 + 1e-6
    for n in whole:
        if n in ("idx", "counts", "z"):
            np.testing.assert_array_equal(few[n], whole[n], err_msg=n)
        else:
            np.testing.assert_allclose(few[n], whole[n], rtol=tol, atol=2e-6, err_msg=n)
    # tokens whose logits are numbers, against the oracle (the first experts of equal score are taken)
    with np.errstate(all="ignore"):
        ref = O.route(f64(to_np(x.float())), f64(to_np(W)), 1.0, 1.0, 1e-6, k, f64(b), mode=mode)
    ok = np.isfinite(ref["z"]).all(1) if kind != "masked" or mode == "norm" else np.ones(T, bool)
    assert ok.sum() == (0 if kind in ("infinite", "nan") or (kind, mode) == ("masked", "norm") else T - 2 * (kind != "masked"))
    np.testing.assert_array_equal(whole["idx"][ok], ref["idx"][ok])
    np.testing.assert_allclose(whole["gate"][ok], ref["g"][ok], rtol=1e-5, atol=1e-6)
    ctx.check_status()
    ctx.close()


@pytest.mark.parametrize("T", [1, 33, 300, 513])
@pytest.mark.parametrize("shift", [0, 1])
def test_prepared_weights_are_a_copy(T, shift):
    """What unipool_router_prepare was given counts until it is called again, whichever router takes the call; weights that
    were not prepared count as they are."""
    M, d, L = 40, 192, 3
    ctx = B.Context(B.make_config(d, 64, M, 2, L, 513, B.BF16, 1e-6, 2.0))
    g = torch.Generator(device="cuda").manual_seed(T)
    W = torch.zeros(L * M * d + shift, device="cuda")[shift:].view(L, M, d).normal_(0, 0.02, generator=g)
    x = torch.randn(T, d, device="cuda", generator=g).bfloat16()
    first = W.clone()
    z = lambda w: x.double() @ w.double().T
    near = lambda out, w: np.abs(out["z"] - to_np(z(w))).max() < 1e-5 * np.abs(out["z"]).max()
    ctx.router_prepare(W, L, M)
    W.normal_(0, 0.02, generator=g)
    for l in range(L):
        assert near(route(ctx, x, W[l], None, 2), first[l])
    ctx.router_prepare(W, L, M)
    assert near(route(ctx, x, W[2], None, 2), W[2])
    ctx.router_prepare(None, 0, M)
    W.copy_(first)
    assert near(route(ctx, x, W[1], None, 2), first[1])
    ctx.close()


def test_weights_of_a_stack_pass_stay_prepared():
    """After a pass through a stack, calls for its routers work with the weights of that pass (without a copy of them: from their
    terms), a later pass with the weights as they are then; also when a call that reads the copy came in between."""
    from paper_2605_06665_b200.stack import UniPoolStack
    T, M, d = 33, 24, 128
    st = UniPoolStack(2, d, 64, M, 2, T, "bf16", c=2.0)
    g = torch.Generator(device="cuda").manual_seed(9)
    for t in (st.W_gu, st.W_down, st.W_r):
        t.normal_(0, 0.05, generator=g)
    x = torch.randn(T, d, device="cuda", generator=g).bfloat16()
    near = lambda z, w: np.abs(to_np(z) - to_np(x.double() @ w.double().T)).max() < 1e-5 * np.abs(to_np(z)).max()
    for copied in (False, True, True):
        if copied:                                             # read the copy once: from then on every pass keeps one
            st.ctx.router_prepare(st.W_r, 2, M)
            route(st.ctx, x, st.W_r[0], None, 2)
        st.forward(x)
        assert near(st.z[0], st.W_r[0])
        old = st.W_r.clone()
        st.W_r.normal_(0, 0.05, generator=g)
        ctx_z = route(st.ctx, x, st.W_r[0], None, 2)["z"]
        assert near(torch.from_numpy(ctx_z), old[0])
        st.forward(x)
        assert near(st.z[0], st.W_r[0])
    st.close()
