"""The stack's public calls in the forms that its own step does not use: layer by layer, with arrays of the
caller's, on small batches.  Each against the path that the parity tests compare with the oracle."""
import pytest

pytestmark = pytest.mark.gpu


def make(L, d, f, M, k, T, dtype="bf16", private=0, seed=0, **kw):
    import torch
    from paper_2605_06665_b200.stack import UniPoolStack
    st = UniPoolStack(L, d, f, M, k, T, dtype, private, c=2.0, **kw)
    g = torch.Generator(device="cuda").manual_seed(seed)
    for w in (st.W_gu, st.W_down, st.W_r):
        w.normal_(0, 0.05, generator=g)
    x0, up = (torch.empty(T, d, device="cuda").normal_(generator=g).to(st.tdtype) for _ in range(2))
    return st, x0, up


@pytest.mark.parametrize("f", [64, 1088])                         # dgrad down on the token-major and the weights-on-M kernels
def test_backward_layer_leaves_operands_for_a_padded_weight_gradient(f):
    """A weight gradient over the padded groups after backward_layer: what the pad rows of dYp and dGU held before
    must not count.  Same sums as the step's own pass, which leaves the padding out: equal, bit for bit."""
    import torch
    from paper_2605_06665_b200 import binding as B
    L, M = 3, 8
    st, x0, up = make(L, 128, f, M, 2, 600, deferred_wgrad=True)
    st.step(x0, up, accumulate=False)
    want = [t.clone() for t in (st.dW_gu, st.dW_down, st.dx[L % 2])]
    for t in (st.dYp, st.dGU):
        t.fill_(float("nan"))
    st.zero_router_grad()
    dx = up
    for l in reversed(range(L)):
        out = torch.empty_like(dx)
        st.backward_layer(l, dx, out)
        dx = out
    st.ctx.pool_wgrad(L, st.cap, st.offsets, st.Xp, st.A, st.dYp, st.dGU, 0, M, st.dW_gu, st.dW_down, B.WGRAD_OVERWRITE)
    torch.cuda.synchronize()
    st.ctx.check_status()
    for got, ref in zip((st.dW_gu, st.dW_down, dx), want):
        assert torch.equal(got, ref)
    st.close()


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_backward_after_a_permute_without_group_sizes(dtype):
    """A caller re-routes tokens and permutes them through the context, without the stack's array of group sizes: the
    backward pass counts the groups itself.  Same result, bit for bit, as with the sizes of that permute."""
    import torch
    L, M, T, k = 2, 9, 700, 2
    got = []
    for with_rows in (True, False):
        st, x0, up = make(L, 128, 192, M, k, T, dtype, deferred_wgrad=True)
        st.forward(x0)                                            # leaves other sizes behind
        idx = torch.randint(0, M, (L, T, 1), generator=torch.Generator().manual_seed(1), dtype=torch.int32)
        st.idx.copy_(torch.cat([idx, (idx + 1) % M], 2))
        st.rows.fill_(3) if not with_rows else None
        for l in range(L):
            c = st.ctx
            rows = st.rows[l] if with_rows else None
            c.dispatch(st.x[l], T, st.idx[l], M, st.offsets[l], st.row_of[l], st.token_of[l], st.tile_expert[l], st.Xp[l], rows)
            c.expert_fwd(st.Xp[l], st.offsets[l], st.tile_expert[l], st.W_gu, st.W_down, 0, M, st.GU[l], st.A[l], st.Yp[l], rows)
            c.combine(st.Yp[l], st.row_of[l], st.gate[l], T, st.x[l], st.x[l + 1])
        st.aux_loss()
        st.zero_router_grad()
        dx = st.backward(up, accumulate=False)
        torch.cuda.synchronize()
        st.ctx.check_status()
        assert (st.rows.cpu() == torch.stack([st.idx[l].flatten().bincount(minlength=M) for l in range(L)]).cpu()).all()
        got.append([t.clone() for t in (dx, st.dW_gu, st.dW_down, st.dW_r)])
        st.close()
    for a, b in zip(*got):
        assert a.isfinite().all()
        if a.shape == (L, M, 128):                                # dW_r: blocks of tokens add with atomics, in any order
            assert (a - b).abs().max() <= 1e-5 * b.abs().max()
        else:
            assert torch.equal(a, b)


def test_fp32_expert_ffn_with_unaligned_results_beside_aligned_operands():
    """fp32 mode: GU, A and dGU that are not 16-byte aligned, with Xp, dYp and weights that are.  Scalar accesses, the
    same sums: equal to the aligned buffers', bit for bit."""
    import torch
    from paper_2605_06665_b200 import binding as B
    d, f, M, T = 64, 128, 5, 400
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *s: torch.empty(*s, device="cuda").normal_(0, 0.1, generator=g)
    x, dy, Wgu, Wd, gate = rnd(T, d), rnd(T, d), rnd(M, 2 * f, d), rnd(M, d, f), rnd(T, 1)
    idx = torch.randint(0, M, (T, 1), device="cuda", generator=g, dtype=torch.int32)
    out = []
    for shift in (0, 1):
        ctx = B.Context(B.make_config(d, f, M, 1, 1, T, B.FP32, 1e-6, 2.0))
        cap = ctx.row_capacity
        new = lambda w: torch.zeros(cap * w + 4, device="cuda")[shift:shift + cap * w].view(cap, w)
        i32 = dict(dtype=torch.int32, device="cuda")
        off, row_of, tok, te, rows = (torch.empty(s, **i32) for s in ((M + 1,), (T, 1), (cap,), (cap // 128,), (M,)))
        Xp, Yp, dYp = (torch.zeros(cap, d, device="cuda") for _ in range(3))
        GU, A, dGU, dx, dgate = new(2 * f), new(f), new(2 * f), torch.empty(T, d, device="cuda"), torch.empty(T, 1, device="cuda")
        dWgu, dWd = torch.empty_like(Wgu), torch.empty_like(Wd)
        ctx.dispatch(x, T, idx, M, off, row_of, tok, te, Xp, rows)
        ctx.expert_fwd(Xp, off, te, Wgu, Wd, 0, M, GU, A, Yp, rows)
        ctx.expert_bwd(dy, T, row_of, gate, tok, off, te, Xp, GU, A, Yp, Wgu, Wd, 0, M, None, dYp, dGU, dx, dgate, dWgu, dWd,
                       B.WGRAD_OVERWRITE, rows)
        torch.cuda.synchronize()
        ctx.check_status()
        ctx.close()
        assert (GU.data_ptr() % 16 != 0) == bool(shift)
        out.append((GU, A, Yp, dGU, dx, dWgu, dWd))
    for a, b in zip(*out):
        assert a.abs().max() > 0 and torch.equal(a, b)


def test_previous_fractions_are_taken_per_group():
    """f-bar of the previous micro-batch: one row per sharing group, dense or not; too few are refused."""
    import torch
    L, G, M = 4, 2, 16
    st, x0, _ = make(L, 64, 64, M, 2, 200, groups=G)
    st.forward(x0)
    prev = torch.rand(G, M // G, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    want = []
    for g in range(G):                                            # the call of one group
        loss, coef, fbar = torch.empty(1, device="cuda"), torch.empty(M // G, device="cuda"), torch.empty(M // G, device="cuda")
        l = slice(g * st.Lg, (g + 1) * st.Lg)
        st.ctx.pool_aux_loss(st.counts[l], st.score_sum[l], st.Lg, st.m, st.T, st.alpha, prev[g].contiguous(), loss, coef, fbar)
        want.append((loss, coef))
    wide = torch.cat([prev, prev + 1], 1)
    for form in (prev, prev.T.contiguous().T, wide[:, :M // G], wide, torch.cat([prev, prev]), prev.double(), prev.cpu()):
        st.loss.fill_(-1)
        st.aux_loss(fbar_prev=form)
        for g, (loss, coef) in enumerate(want):
            assert torch.equal(st.loss[g:g + 1], loss) and torch.equal(st.coef[g], coef)
    for bad in (prev[0], prev[:1], prev[:, :4], prev.flatten()):
        with pytest.raises(IndexError):
            st.aux_loss(fbar_prev=bad)
    st.close()


NAMES = ("x", "dx", "loss", "idx", "gate", "z", "dW_gu", "dW_down", "dW_r", "dsigma")


def same(got, want, other_order=("dW_r",)):
    """Equal bit for bit, but for sums that are taken in another order: dW_r always (its blocks add with atomics), fp32
    sums of some hundred terms, random signs: 1e-5 of the largest value."""
    import torch
    for n, a, w in zip(NAMES, got, want):
        if n in other_order:
            assert (a.double() - w.double()).abs().max() <= 1e-5 * w.double().abs().max(), n
        else:
            assert torch.equal(a, w), n


def stack_results(st, x0, up):
    import torch
    dx = st.step(x0, up, accumulate=False)
    torch.cuda.synchronize()
    st.ctx.check_status()
    return [t.clone() for t in (st.x[st.L], dx, st.loss, st.idx, st.gate, st.z, st.dW_gu, st.dW_down, st.dW_r, st.dsigma)]


BIAS_FORMS = dict(
    expanded=lambda b: b[0].expand(*b.shape), list=list, tuple_with_none=lambda b: (None,) + tuple(b[1:]),
    transposed=lambda b: b.T.contiguous().T, slice_of_a_wider=lambda b: b.repeat(1, 2)[:, :b.shape[1]],
    double=lambda b: b.double(), host=lambda b: b.cpu())


@pytest.mark.parametrize("form", sorted(BIAS_FORMS))
@pytest.mark.parametrize("kw", [dict(deferred_wgrad=True), dict(recompute=True), dict(dtype="fp32")])
def test_bias_in_other_forms_than_one_dense_array(form, kw):
    """A bias whose layers are not the rows of one dense float array gives what the dense array of the same values gives."""
    import torch
    L, M = 3, 10
    st, x0, up = make(L, 64, 128, M, 2, 150, **kw)
    b = torch.empty(L, M, device="cuda").normal_(generator=torch.Generator(device="cuda").manual_seed(1))
    given = BIAS_FORMS[form](b)
    st.bias = torch.stack([torch.zeros(M, device="cuda") if v is None else v.cuda().float() for v in given])
    want = stack_results(st, x0, up)
    st.bias = given
    got = stack_results(st, x0, up)
    # recompute: layer by layer instead of in runs of layers; fp32: whole groups instead of their tokens
    same(got, want, ("dW_r", "dW_gu", "dW_down") if "recompute" in kw or "dtype" in kw else ("dW_r",))
    st.bias = [b[0, :4]] * L
    with pytest.raises(ValueError):
        st.forward(x0)
    st.close()


def test_arrays_of_the_caller_that_are_slices_of_larger_ones():
    """Activations, logits and gradients that the caller keeps in padded arrays of its own; too few scales are refused."""
    import torch
    L, M, d, T = 3, 8, 64, 150
    st, x0, up = make(L, d, 128, M, 2, T, deferred_wgrad=True)
    want = stack_results(st, x0, up)
    st.dW_r = torch.zeros(L, M + 2, d, device="cuda")[:, :M]
    st.z = torch.zeros(L, T + 1, M, device="cuda")[:, :T]
    st.x = torch.zeros(L + 1, T + 8, d, dtype=st.tdtype, device="cuda")[:, :T]
    same(stack_results(st, x0, up), want)
    st.znorm = list(torch.zeros(L, T, device="cuda"))             # an array per layer
    same(stack_results(st, x0, up), want)
    st.sigma = st.sigma[:2]
    with pytest.raises(IndexError):
        st.forward(x0)
    st.close()


def test_recompute_holds_as_few_layers_as_asked_or_as_fit():
    """wgrad_layers=1 is one shared slot for every permuted array; the default holds more layers, and one where more do
    not fit the device."""
    import torch
    shape = (8, 512, 1024, 128, 1, 128)

    def build(**kw):
        torch.cuda.empty_cache()
        return make(*shape, recompute=True, **kw)

    def slots(st):
        return [getattr(st, n).shape[0] for n in ("Xp", "A", "dYp", "dGU", "GU", "Yp")]

    torch.cuda.empty_cache()
    before = torch.cuda.memory_reserved()
    st, x0, up = build(wgrad_layers=1)
    need = torch.cuda.memory_reserved() - before
    assert slots(st) == [1] * 6
    want = stack_results(st, x0, up)
    st.close()
    del st
    st, x0, up = build()
    assert slots(st) == [4, 4, 4, 4, 1, 1]
    same(stack_results(st, x0, up), want, ("dW_r", "dW_gu", "dW_down"))
    st.close()
    del st
    torch.cuda.empty_cache()
    limit = torch.cuda.memory_reserved() + need + 200e6                          # four layers need 400 MB more than one
    torch.cuda.set_per_process_memory_fraction(limit / torch.cuda.get_device_properties(0).total_memory)
    try:
        with pytest.raises(torch.OutOfMemoryError):
            build(wgrad_layers=4)
        st, x0, up = build()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert slots(st) == [1] * 6
    same(stack_results(st, x0, up), want, ("dW_r", "dW_gu", "dW_down"))
    st.close()
    for kw in (dict(recompute=True, wgrad_layers=0), dict(recompute=True, wgrad_layers=9), dict(wgrad_layers=2)):
        with pytest.raises(ValueError):
            make(*shape, **kw)


def test_an_expired_wait_of_one_lane_is_known_to_its_warp():
    """Warps that act as one wait as one: when a lane's wait gives up, all 32 have its answer."""
    import torch
    from paper_2605_06665_b200 import binding as B
    ctx = B.Context(B.make_config(64, 64, 8, 1, 1, 64, B.BF16, 1e-6, 1.0))
    ctx.selftest_wait(20_000)
    torch.cuda.synchronize()
    with pytest.raises(B.UniPoolError, match="site 99, detail 32"):
        ctx.check_status()
    ctx.check_status()
    ctx.close()


def test_host_threads_with_contexts_of_different_sizes():
    """Launches of the same kernels with few and many experts from two threads: neither is refused for the shared memory
    that the other asked for (before, one thread could lower the function's limit between another's call and launch)."""
    import threading
    import torch
    L, d, f, T = 300, 256, 1600, 64                               # many layers: the threads meet inside the native loop
    stacks = [make(L, d, f, M, 1, T, recompute=True) for M in (4, 300)]           # the weights-on-M kernels and the router
    [st.W_down.mul_(1e-3) for st, _, _ in stacks]                 # so that 300 residual layers stay finite
    want = [st.forward(x0).clone() for st, x0, _ in stacks]
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            st, x0, _ = stacks[i]
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(20):
                    st.forward(x0)
                torch.cuda.current_stream().synchronize()
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    torch.cuda.synchronize()
    assert not errors
    for (st, _, _), w in zip(stacks, want):
        st.ctx.check_status()
        assert torch.equal(st.x[L], w)
        st.close()


@pytest.mark.parametrize("shape,kw", [
    ((3, 64, 128, 9, 2, 300), dict(deferred_wgrad=True)),
    ((3, 64, 128, 9, 2, 300), {}),
    ((3, 128, 192, 9, 2, 300), dict(dtype="fp32", deferred_wgrad=True)),
    ((4, 64, 128, 16, 2, 300), dict(groups=2, deferred_wgrad=True)),
    ((3, 64, 128, 24, 1, 300), dict(private=8, router="softmax")),
    ((5, 256, 384, 48, 1, 40), dict(recompute=True)),             # runs of two, two and one layer
    ((5, 256, 384, 48, 1, 40), dict(recompute=True, wgrad_layers=1)),
    ((2, 768, 2048, 96, 2, 16384), dict(deferred_wgrad=True)),    # the sizes that the oracle checks layer by layer
    ((2, 768, 2048, 16, 2, 16384), dict(private=8)),
    ((2, 768, 512, 384, 8, 16384), dict(deferred_wgrad=True)),
    ((2, 1536, 4096, 192, 2, 32768), dict(recompute=True)),
])
def test_native_loops_give_what_the_layers_give_one_by_one(shape, kw):
    """forward, aux_loss and backward against the same calls layer by layer, which the parity tests compare with the
    oracle: every array equal, bit for bit, but for sums in another order (weight gradients of recomputed runs of layers;
    fp32: of whole groups instead of their tokens)."""
    import torch
    L = shape[0]
    st, x0, up = make(*shape, **kw)
    state = ("x", "idx", "gate", "counts", "score_sum", "znorm", "z", "offsets", "row_of", "token_of", "tile_expert", "loss",
             "coef", "fbar", "dgate")
    both = []
    for native in (True, False):
        st.zero_grad()
        if native:
            dx = st.step(x0, up)
        else:
            st.ctx.router_prepare(st.W_r, L, st.m)
            st.x[0].copy_(x0)
            for l in range(L):
                st.forward_layer(l)
            for g in range(st.G):
                l = slice(g * st.Lg, (g + 1) * st.Lg)
                st.ctx.pool_aux_loss(st.counts[l], st.score_sum[l], st.Lg, st.m, st.T, st.alpha, None, st.loss[g:g + 1],
                                     st.coef[g], st.fbar[g])
            dx = up
            for l in reversed(range(L)):
                out = torch.empty_like(up)
                st.backward_layer(l, dx, out)
                dx = out
            for g in range(st.G if st.deferred_wgrad else 0):
                l = g * st.Lg
                st.ctx.pool_wgrad(st.Lg, st.cap, st.offsets[l:], st.Xp[l:], st.A[l:], st.dYp[l:], st.dGU[l:], g * st.m, st.m,
                                  st.dW_gu, st.dW_down)
        torch.cuda.synchronize()
        st.ctx.check_status()
        both.append({n: getattr(st, n).clone() for n in state + ("dW_r", "dsigma", "dW_gu", "dW_down")} | dict(dx=dx.clone()))
        for n in state:
            getattr(st, n).zero_()
    got, want = both
    other_order = {"dW_r"} | ({"dW_gu", "dW_down"} if st.nw > 1 or "dtype" in kw else set())
    for n in want:
        if n in other_order:
            assert (got[n] - want[n]).abs().max() <= 1e-5 * want[n].abs().max(), n
        else:
            assert torch.equal(got[n], want[n]), n
    st.close()
    del st, both, got, want
    torch.cuda.empty_cache()


def test_evaluation_without_the_arrays_of_backward():
    """A stack that only evaluates may give up what backward needs; a backward call then is refused, not run."""
    import torch
    from paper_2605_06665_b200 import binding as B
    st, x0, up = make(2, 64, 128, 8, 2, 150, deferred_wgrad=True)
    want = st.forward(x0).clone()
    loss = st.aux_loss().clone()
    for n in ("dYp", "dGU", "dx", "dW_gu", "dW_down"):
        setattr(st, n, None)
    assert torch.equal(st.forward(x0), want) and torch.equal(st.aux_loss(), loss)
    st.dx = torch.empty(2, st.T, st.d, dtype=st.tdtype, device="cuda")
    with pytest.raises(B.UniPoolError):
        st.backward(up)
    torch.cuda.synchronize()
    st.ctx.check_status()
    st.close()
