"""The torch.autograd glue: loss.backward() through csat_attention gives csat_backward's gradients."""
import numpy as np
import pytest
import torch

from oracle import csat_oracle as orc
from paper_2507_02957_b200 import binding, workloads as wl
from gpu_util import TOL, device_inputs, make_ctx, rel_err, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("save", [True, False], ids=["saving_forward", "recomputing_backward"])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_autograd_function_matches_the_library_and_the_oracle(dtype, save):
    from paper_2507_02957_b200.autograd import csat_attention
    w = wl.shrink(wl.CONFIGS["c2"], B=2, H=2, n_q=150, lam=0.0) if dtype == "bf16" else wl.shrink(wl.CONFIGS["c1"], B=2, H=2, n=100, n_q=37, m=40, d=32, T=3, lam=0.0)
    inp = wl.make_inputs(w)
    Q, K, V, _ = device_inputs(w, inp)
    ctx = make_ctx(w)
    q, k, v = (t.clone().requires_grad_(True) for t in (Q, K, V))
    out = csat_attention(ctx, q, k, v, save_for_backward=save)
    G = torch.randn(out.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3)).to(out.dtype)
    (out.float() * G.float()).sum().backward()
    # the same numbers as the library's own calls
    binding.csat_set_i64(ctx.h, binding.CSAT_SAVE_FOR_BACKWARD, 0)
    assert torch.equal(out.detach(), ctx.forward(Q, K, V)) or rel_err(to_np(out.detach()), to_np(ctx.forward(Q, K, V))) <= TOL[dtype]
    dQ, dK, dV = ctx.backward(Q, K, V, G)
    for a, b in zip((q.grad, k.grad, v.grad), (dQ, dK, dV)):
        assert torch.equal(a, b)
    # and the oracle's (lambda = 0: every shrinkage decision is |x| > 0 on both sides)
    ref = orc.csat_backward(inp["Q"], inp["K"], inp["V"], to_np(ctx.get_phi()), to_np(G), T=w.T, lam=0.0)
    for g, rf in zip((q.grad, k.grad, v.grad), ref):
        assert rel_err(to_np(g), rf) <= (2e-2 if dtype == "bf16" else 2e-5)
    ctx.close()


def test_module_owns_a_context():
    from paper_2507_02957_b200.autograd import CsatAttention
    mod = CsatAttention(256, 64, 64, 2, B=1, T=4, lam=0.01, seed=5)
    g = torch.Generator(device="cuda").manual_seed(1)
    Q, K, V = ((torch.randn(1, 2, 256, 64, device="cuda", generator=g) / 8).bfloat16().requires_grad_(True) for _ in range(3))
    out = mod(Q, K, V)
    assert out.shape == (1, 2, 256, 64) and torch.isfinite(out).all()
    out.float().sum().backward()
    assert all(t.grad is not None and torch.isfinite(t.grad).all() for t in (Q, K, V))


@pytest.mark.parametrize("dtype,d,profile", [("fp32", 32, 0), ("fp32", 64, 0), ("bf16", 64, 4), ("bf16", 128, 4), ("bf16", 64, 0), ("bf16", 96, 0)])
def test_other_calls_between_a_forward_and_its_backward(dtype, d, profile):
    """Whatever else the context computes in between, on other data, the gradients are those of the forward's own tensors, bit for
    bit as without saved state."""
    from paper_2507_02957_b200.autograd import csat_attention
    B, H, n, nq, m, T = 2, 3, 143, 90, 72 if d < 96 else 130, 4
    g = torch.Generator(device="cuda").manual_seed(d)
    ctx = binding.Csat(n, m, d, H, 3, B=B, n_q=nq, dtype=dtype, T=T, lam=0.02)
    binding.csat_set_i64(ctx.h, binding.CSAT_PROFILE, profile)
    Q, K, V, G, Q2, K2, V2 = (torch.randn(B, H, r, d, generator=g, device="cuda").to(ctx.torch_dtype) for r in (nq, n, n, nq, nq, n, n))
    want = ctx.backward(Q, K, V, G)
    host = [t.cpu() for t in (Q2, K2, V2, Q2)]
    between = {"forward_host": lambda: ctx.forward_host(*host), "forward": lambda: ctx.forward(Q2, K2, V2), "attend": lambda: ctx.attend(Q2),
               "compress": lambda: ctx.reduce_partials(torch.stack([ctx.compress_partial(K2[:, :, :80].contiguous(), V2[:, :, :80].contiguous(), 0)])),
               "none": lambda: None}
    for name, call in between.items():
        leaves = [t.clone().requires_grad_(True) for t in (Q, K, V)]
        out = csat_attention(ctx, *leaves)
        call()
        grads = torch.autograd.grad(out, leaves, G)
        assert all(torch.equal(a, b) for a, b in zip(grads, want)), name
    ctx.close()


@pytest.mark.parametrize("dtype,d", [("fp32", 32), ("bf16", 64), ("bf16", 128)])
def test_nothing_is_recorded_where_no_gradient_can_be_asked_for(dtype, d):
    """Without gradients (or inputs that require none) csat_attention is Csat.forward: the same bits, no scratch of the backward."""
    from paper_2507_02957_b200.autograd import CsatAttention
    mod = CsatAttention(256, 130, d, 2, B=2, n_q=70, T=4, lam=0.01, seed=5, dtype=dtype)
    g = torch.Generator(device="cuda").manual_seed(1)
    Q, K, V = (torch.randn(2, 2, r, d, device="cuda", generator=g).to(mod.csat.torch_dtype) for r in (70, 256, 256))
    want, before = mod.csat.forward(Q, K, V), mod.csat.workspace_bytes
    leaves = [t.clone().requires_grad_(True) for t in (Q, K, V)]
    with torch.no_grad():
        assert torch.equal(mod(*leaves), want)
    assert torch.equal(mod(Q, K, V), want) and mod.csat.workspace_bytes == before
    out = mod(Q, leaves[1], V)                              # one of them is enough
    assert mod.csat.workspace_bytes > before
    with torch.no_grad():                                   # and a call without gradients takes nothing from it
        mod(Q, K, V)
    G = torch.randn(out.shape, device="cuda", generator=g).to(out.dtype)
    dK, = torch.autograd.grad(out, leaves[1:2], G)
    binding.csat_set_i64(mod.csat.h, binding.CSAT_SAVE_FOR_BACKWARD, 0)
    assert torch.equal(dK, mod.csat.backward(Q, K, V, G)[1])


@pytest.mark.parametrize("dtype,d", [("fp32", 64), ("bf16", 64), ("bf16", 128)])
def test_direct_calls_beside_csat_attention(dtype, d):
    """The key that csat_attention sets is its own: a direct backward on other tensors does not start from its forward's state, a
    direct forward does not record, and a key set by hand stays as it was set."""
    from paper_2507_02957_b200.autograd import csat_attention
    KEY = binding.CSAT_SAVE_FOR_BACKWARD
    B, H, n, nq, m, T = 2, 3, 143, 90, 130, 4
    g = torch.Generator(device="cuda").manual_seed(d)
    ctx = binding.Csat(n, m, d, H, 3, B=B, n_q=nq, dtype=dtype, T=T, lam=0.02)
    x, y = ([torch.randn(B, H, r, d, generator=g, device="cuda").to(ctx.torch_dtype) for r in (nq, n, n, nq)] for _ in range(2))
    out_y, want_x, want_y = ctx.forward(*y[:3]), ctx.backward(*x), ctx.backward(*y)
    same = lambda got, want: all(torch.equal(a, b) for a, b in zip(got, want))
    leaves = [t.clone().requires_grad_(True) for t in x[:3]]
    for by_hand in (None, 1, 0):
        if by_hand is not None:
            binding.csat_set_i64(ctx.h, KEY, by_hand)
        out = csat_attention(ctx, *leaves)
        assert same(ctx.backward(*y), want_y)
        assert same(torch.autograd.grad(out, leaves, x[3]), want_x)
        out = csat_attention(ctx, *leaves)
        if not by_hand:
            assert torch.equal(ctx.forward(*y[:3]), out_y)
        else:
            ctx.forward(*y[:3])
            assert same(ctx.backward(*y), want_y)
        assert binding.csat_get_i64(ctx.h, KEY) == (by_hand or 0)
        assert same(torch.autograd.grad(out, leaves, x[3]), want_x)
        out = csat_attention(ctx, *leaves)
        binding.csat_set_i64(ctx.h, KEY, 1)
        res = torch.empty_like(y[0])
        binding.csat_forward(ctx.h, *y[:3], res)
        assert same(torch.autograd.grad(out, leaves, x[3]), want_x)
        out = csat_attention(ctx, *leaves)                   # and it still saves: both backwards start from the state
        launches = []
        for _ in range(2):
            assert same(torch.autograd.grad(out, leaves, x[3], retain_graph=True), want_x)
            launches.append(ctx.launches)
        binding.csat_set_i64(ctx.h, KEY, 0)
        ctx.backward(*x)
        assert max(launches) < ctx.launches
    ctx.close()


def test_a_closed_context_is_refused():
    from paper_2507_02957_b200.autograd import csat_attention
    ctx = binding.Csat(140, 70, 64, 2, 3, dtype="fp32", T=2, lam=0.02)
    Q, K, V = (torch.randn(1, 2, 140, 64, device="cuda").requires_grad_(True) for _ in range(3))
    out = csat_attention(ctx, Q, K, V)
    ctx.close()
    for call in (lambda: torch.autograd.grad(out.sum(), (Q, K, V)), lambda: csat_attention(ctx, Q, K, V), lambda: ctx.forward(Q, K, V)):
        with pytest.raises(binding.CsatError):
            call()
