"""GPU tests of the library's behaviour around its compute kernels: the host-buffer forward with more batch
elements than it has pipeline events, and a context whose re-allocation failed."""
import pytest
import torch

from paper_2507_02957_b200 import binding, workloads as wl
from gpu_util import device_inputs, make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H", [(65, 1), (70, 3), (3, 50)])
def test_host_forward_with_more_pairs_than_pipeline_chunks(B, H):
    """The pipelined host-buffer forward cuts the job into at most 64 runs of (batch, head) pairs; with more batch
    elements than that a run spans several of them.  The call must return and equal csat_forward bit for bit."""
    w = wl.Workload("many_pairs", B, H, 128, 96, 64, 64, "bf16", 2, 0.01, "iid", 51)
    inp = wl.make_inputs(w)
    Q, K, V, _ = device_inputs(w, inp)
    ctx = make_ctx(w)
    ref = ctx.forward(Q, K, V).cpu()
    Qh, Kh, Vh = (t.cpu().pin_memory() for t in (Q, K, V))
    oh = torch.full_like(Qh, float("nan")).pin_memory()
    ctx.forward_host(Qh, Kh, Vh, oh)
    assert torch.equal(oh, ref)
    ctx.close()


def test_failed_reallocation_is_refused_until_a_setter_succeeds():
    """A setter whose cudaMalloc fails must not leave a context that launches kernels on null buffers: compute calls
    and getters answer CSAT_ERR_STATE until a re-allocating setter succeeds.  The failure is injected on the host."""
    w = wl.Workload("realloc", 2, 2, 256, 256, 64, 64, "bf16", 3, 0.01, "iid", 52)
    inp = wl.make_inputs(w)
    Q, K, V, _ = device_inputs(w, inp)
    ctx = make_ctx(w)
    ref = ctx.forward(Q, K, V).clone()
    lib = binding.load()
    s = torch.cuda.current_stream().cuda_stream
    out = torch.empty_like(Q)
    for key, bad_value, good_value in [(binding.CSAT_BATCH, 5, 2), (binding.CSAT_SEPARATE_PHI, 1, 0),
                                       (binding.CSAT_DTYPE, binding.CSAT_DTYPE_FP32, binding.CSAT_DTYPE_BF16)]:
        for countdown in (1, 2):
            assert binding.csat_debug_fail_alloc(countdown) == 0
            rc = lib.csat_set_i64(ctx.h, key, bad_value)
            binding.csat_debug_fail_alloc(0)
            if key == binding.CSAT_BATCH and countdown == 2:
                assert rc == 0                                        # that setter allocates once: nothing failed
            else:
                assert rc == 3, (key, countdown, rc)                  # CSAT_ERR_ALLOC
                assert lib.csat_forward(ctx.h, Q.data_ptr(), K.data_ptr(), V.data_ptr(), out.data_ptr(), s) == 6
                assert "re-allocate" in binding.csat_last_error(ctx.h)
                phi = torch.empty(2 * w.H, w.m, w.n, dtype=torch.float32, device="cuda")
                assert lib.csat_get_phi(ctx.h, phi.data_ptr(), s) == 6
                assert lib.csat_backward(ctx.h, *(t.data_ptr() for t in (Q, K, V, Q, out, out, out)), s) == 6
            binding.csat_set_i64(ctx.h, key, good_value)              # succeeds and repairs the context
            torch.cuda.synchronize()
            assert torch.equal(ctx.forward(Q, K, V), ref), (key, countdown)
    ctx.close()


@pytest.mark.parametrize("shape", [(1, 3, 131, 67, 64, 67), (2, 2, 203, 37, 128, 139), (3, 1, 392, 200, 64, 200),
                                   (1, 2, 100, 50, 40, 41)])
@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_workspace_canary_finds_no_unwritten_row(shape, dtype):
    """CSAT_DEBUG_CANARY fills the K~|V~ workspace with NaN before every compression: on ragged shapes (measurement and
    token counts that are no multiples of the tiles, odd batches, both kernel families) the forward and the backward
    must stay finite and give the same bits as without the canary, i.e. every workspace row that is read was
    written by the same call."""
    B, H, n, nq, d, m = shape
    w = wl.Workload("canary", B, H, n, nq, d, m, dtype, 3, 0.01, "iid", 57)
    inp = wl.make_inputs(w)
    Q, K, V, _ = device_inputs(w, inp)
    ctx = make_ctx(w)
    ref = ctx.forward(Q, K, V).clone()
    G = torch.randn_like(Q)
    gref = [t.clone() for t in ctx.backward(Q, K, V, G)]
    binding.csat_set_i64(ctx.h, binding.CSAT_DEBUG_CANARY, 1)
    assert binding.csat_get_i64(ctx.h, binding.CSAT_DEBUG_CANARY) == 1
    out = ctx.forward(Q, K, V)
    assert torch.isfinite(out).all() and torch.equal(out, ref)
    for a, b in zip(ctx.backward(Q, K, V, G), gref):
        assert torch.isfinite(a).all() and torch.equal(a, b)
    ctx.close()


@pytest.mark.parametrize("first", ["saving_forward", "backward"])
def test_a_saving_float32_forward_without_memory_for_its_state(first):
    """The allocation fails (on the host) where the state is asked for with the rest of the scratch, or for itself behind an earlier
    backward: the forward returns what it returns, the backward recomputes, nothing is asked for again until the key changes, and
    the earlier backward's decisions stay."""
    B, H, n, nq, d, m, T = 2, 3, 140, 70, 40, 60, 4
    g = torch.Generator(device="cuda").manual_seed(4)
    Q, K, V, G = (torch.randn(B, H, r, d, generator=g, device="cuda") for r in (nq, n, n, nq))
    SAVE = binding.CSAT_SAVE_FOR_BACKWARD
    plain, ctx = (binding.Csat(n, m, d, H, 3, B=B, n_q=nq, dtype="fp32", T=T, lam=0.02) for _ in range(2))
    for c in (plain, ctx):
        binding.csat_set_i64(c.h, binding.CSAT_KEEP_MASKS, 1)
    out, want = plain.forward(Q, K, V), plain.backward(Q, K, V, G)
    masks = plain.backward_masks()
    if first == "backward":
        ctx.backward(Q, K, V, G)
    binding.csat_set_i64(ctx.h, SAVE, 1)
    # (with CSAT_KEEP_MASKS the scratch begins with the decisions: its second allocation is the one the state is in)
    binding.csat_debug_fail_alloc(2 if first == "saving_forward" else 1)
    for _ in range(2):                                       # the second one would succeed if it asked
        assert torch.equal(ctx.forward(Q, K, V), out)
        binding.csat_debug_fail_alloc(0)
        assert ctx.workspace_bytes == plain.workspace_bytes
        if first == "backward":
            assert torch.equal(ctx.backward_masks(), masks)
        assert all(torch.equal(a, b) for a, b in zip(ctx.backward(Q, K, V, G), want)) and ctx.launches > 3
    binding.csat_set_i64(ctx.h, SAVE, 0)
    binding.csat_set_i64(ctx.h, SAVE, 1)
    ctx.forward(Q, K, V)
    assert torch.equal(ctx.backward_masks(), masks)
    assert ctx.workspace_bytes > plain.workspace_bytes
    assert all(torch.equal(a, b) for a, b in zip(ctx.backward(Q, K, V, G), want)) and ctx.launches == 3
    assert torch.equal(ctx.backward_masks(), masks)
    for c in (plain, ctx):
        c.close()


@pytest.mark.parametrize("d", [40, 64, 96, 120])
def test_a_context_holds_what_its_storage_type_needs(d):
    """Phi, K~|V~ (bf16 with V~ B behind it), the decoder in float32 and float64 and its bf16 operands; the operands in two parts
    only where a kernel reads them, also after the storage type has changed."""
    B, H, n, m = 2, 3, 200, 130
    n_pad = -(-n // 64) * 64
    Q, K, V = (torch.randn(B, H, n, d, generator=torch.Generator(device="cuda").manual_seed(i), device="cuda") for i in range(3))
    ctx = binding.Csat(n, m, d, H, 3, B=B, dtype="fp32", T=3, lam=0.02)
    outs = {}
    for dtype, es, code in (("fp32", 4, binding.CSAT_DTYPE_FP32), ("bf16", 2, binding.CSAT_DTYPE_BF16)) * 2:
        binding.csat_set_i64(ctx.h, binding.CSAT_DTYPE, code)
        two_parts = dtype == "bf16" and d <= 96 and d != 64
        decoder = H * d * d * (2 * 8 + 3 * 4 + (3 + (6 if two_parts else 0)) * 2) + 2 * H * 4
        assert ctx.workspace_bytes == H * m * n_pad * es + B * H * m * (3 if dtype == "bf16" else 2) * d * es + decoder
        ctx.torch_dtype = torch.bfloat16 if dtype == "bf16" else torch.float32
        out = ctx.forward(*(t.to(ctx.torch_dtype) for t in (Q, K, V)))
        assert torch.equal(out, outs.setdefault(dtype, out)) and torch.isfinite(out).all()
    ctx.close()
    if d in (40, 96):                                        # the added allocation fails: refused until it succeeds
        ctx = binding.Csat(n, m, d, H, 3, B=B, dtype="fp32", T=3, lam=0.02)
        binding.csat_debug_fail_alloc(1)
        with pytest.raises(binding.CsatError):
            binding.csat_set_i64(ctx.h, binding.CSAT_DTYPE, binding.CSAT_DTYPE_BF16)
        binding.csat_debug_fail_alloc(0)
        ctx.torch_dtype = torch.bfloat16
        with pytest.raises(binding.CsatError):
            ctx.forward(*(t.bfloat16() for t in (Q, K, V)))
        binding.csat_set_i64(ctx.h, binding.CSAT_DTYPE, binding.CSAT_DTYPE_BF16)
        assert torch.equal(ctx.forward(*(t.bfloat16() for t in (Q, K, V))), outs["bf16"])
        ctx.close()
