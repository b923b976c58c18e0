"""The router kernel for few tokens at the edges of its clusters, slices of experts and steps along the width, against the
float64 oracle; one token more is the tensor-core router's."""
import numpy as np
import pytest
import torch

from oracle import unipool_oracle as O
from parity_utils import check_routing, f64, to_np
from paper_2605_06665_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,M,d,k,mode,biased,shift", [
    (1, 96, 768, 2, "norm", False, 0), (7, 33, 64, 3, "norm", True, 0), (8, 4, 128, 1, "softmax", False, 0),
    (9, 509, 192, 8, "norm", False, 0), (33, 96, 768, 8, "softmax", True, 0), (33, 7, 832, 2, "norm", True, 1),
    (232, 40, 320, 2, "norm", False, 0), (233, 41, 320, 2, "softmax", True, 3), (463, 65, 1408, 4, "norm", False, 0),
    (464, 512, 576, 8, "norm", True, 0), (465, 96, 256, 2, "norm", False, 0), (200, 192, 2944, 2, "norm", False, 0),
    (464, 128, 1408, 2, "norm", False, 0), (464, 129, 960, 2, "softmax", False, 0), (233, 129, 1024, 2, "norm", True, 0),
    (233, 128, 1472, 8, "norm", False, 0), (464, 192, 1536, 2, "norm", False, 0), (232, 512, 1408, 2, "softmax", False, 0),
])
def test_route_few_tokens(T, M, d, k, mode, biased, shift):
    """shift: elements by which the weights miss 16-byte alignment (x has to keep it).  The second call finds the accumulators that
    the first one has left.  Sixteen tokens to a cluster (from 233) only while the width does not make the other router the
    faster one for some weights."""
    few = T <= 232 or (T <= 464 and d <= (1408 if M <= 128 else 960))
    rng = np.random.default_rng(T + M)
    ctx = B.Context(B.make_config(d, 64, M, k, 1, max(T, 512), B.BF16, 1e-6, 2.0,
                                  B.ROUTER_SOFTMAX if mode == "softmax" else B.ROUTER_NORM))
    nan = lambda *s, dtype=torch.float32: torch.full(s, float("nan"), device="cuda").to(dtype)
    x = torch.zeros(T * d + 1, dtype=torch.bfloat16, device="cuda")
    x, odd = x[:-1].view(T, d), x[1:].view(T, d)
    W = torch.zeros(M * d + shift, device="cuda")[shift:].view(M, d)
    x.copy_(torch.from_numpy(rng.standard_normal((T, d), dtype=np.float32)))
    W.copy_(torch.from_numpy(0.02 * rng.standard_normal((M, d), dtype=np.float32)))
    bias = torch.from_numpy(rng.standard_normal(M, dtype=np.float32)).cuda() if biased else None
    idx, counts = torch.full((T, k), -7, dtype=torch.int32, device="cuda"), torch.zeros(M, dtype=torch.int32, device="cuda")
    gate, S, n, z = nan(T, k), nan(M), nan(T), nan(T, M)
    with pytest.raises(RuntimeError, match="aligned"):
        ctx.route(odd, T, W, 0.7, bias, M, idx, gate, counts, S, n, z)
    ctx.profile_enable(True)
    for _ in range(2):
        ctx.route(x, T, W, 0.7, bias, M, idx, gate, counts, S, n, z)
    assert ctx.profile_read()["route_logits"][1] == (0 if few else 2)        # the other router splits the weights
    ctx.profile_enable(False)
    args = (f64(to_np(x.float())), f64(to_np(W)), 0.7, 2.0, 1e-6, k, None if bias is None else f64(to_np(bias)))
    ref = O.route(*args, mode=mode)
    check_routing(to_np(idx), ref["z"], ref["idx"], k, mode=mode)
    ref = O.route(*args, forced_idx=to_np(idx), mode=mode)
    scale = np.abs(ref["z"]).max()
    # fp32 sums of d terms: errors of some sqrt(d) 2^-24 of the terms' norm, 1e-5 at d = 3000 with room for the largest
    assert np.abs(to_np(z) - ref["z"]).max() / scale < 1e-5
    for got, want in ((n, "n"), (gate, "g"), (S, "S")):
        assert np.abs(f64(to_np(got)) - ref[want]).max() / np.abs(ref[want]).max() < 1e-5, want
    assert (to_np(counts) == ref["counts"]).all()
    ctx.check_status()
    ctx.close()
