"""Both routers of the bf16 mode on values out of the ordinary: score sums beyond what their accumulators hold."""
import numpy as np
import pytest
import torch

from parity_utils import to_np
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
