"""bf16, d = 64: the warp-level attention / recovery of small jobs and the tcgen05 kernel behind it at the same edges (query
counts around 16 and 64, measurement counts around a chunk of 64), on either side of the rule that chooses between them
(one CTA of 64 queries per SM), against the float64 oracle; and the backward, whose forward records its decisions in
either kernel."""
import numpy as np
import pytest
import torch

from oracle import csat_oracle as orc
from paper_2507_02957_b200 import binding, workloads as wl
from gpu_util import TOL, device_inputs, make_ctx, rel_err, to_dev, to_np

pytestmark = pytest.mark.gpu
D = 64


def _setup(B, H, nq, m, T, lam):
    w = wl.Workload("warp", B, H, 200, nq, D, m, "bf16", T, lam, "iid", 700 + nq)
    inp = wl.make_inputs(w)
    return w, inp, device_inputs(w, inp)[:3], make_ctx(w)


@pytest.mark.parametrize("nq", [1, 16, 17, 63, 65, 130])
@pytest.mark.parametrize("heads", [(1, 3), (4, 40)], ids=["small", "beyond"])
def test_forward_at_the_edges(heads, nq):
    B, H = heads
    m = 64 if nq % 2 else 131
    w, inp, (Q, K, V), ctx = _setup(B, H, nq, m, 3, 0.01)
    phi = to_np(ctx.get_phi())
    r = np.random.default_rng(nq)
    Psi = wl.round_to_storage((np.eye(D) + 0.3 * r.standard_normal((D, D)) / 8).astype(np.float32), "bf16")
    S = wl.round_to_storage((0.6 * np.eye(D) + 0.4 * r.standard_normal((H, D, D)) / 8).astype(np.float32), "bf16")
    Bm = wl.round_to_storage((r.standard_normal((H, D, D)) / 8).astype(np.float32), "bf16")
    th = (0.02 * r.uniform(0.5, 1.5, size=(3, H))).astype(np.float32)
    th[1, 0] = 0.0

    def check(**kw):
        ref = orc.csat_forward(inp["Q"], inp["K"], inp["V"], phi, **kw)
        out = to_np(ctx.forward(Q, K, V))
        assert np.isfinite(out).all() and np.abs(ref).max() > 0
        assert rel_err(out, ref) <= TOL["bf16"], (heads, nq, list(kw), rel_err(out, ref))

    for T, lam in ((0, 0.0), (1, 0.001), (3, 0.001), (3, 0.0)):
        ctx.set(T=T, lam=lam)
        check(T=T, lam=lam)
    ctx.set_dictionary(to_dev(Psi, "bf16"))
    ctx.set(lam=0.001)
    check(T=3, lam=0.001, Psi=Psi.astype(np.float64))
    # supplied (non-symmetric) weights with one threshold per layer, one of them zero
    ctx.set_lista_weights(to_dev(S, "bf16"), to_dev(Bm, "bf16"), torch.from_numpy(th).cuda())
    check(T=3, lam=0.0, Psi=Psi.astype(np.float64), weights=(S.astype(np.float64), Bm.astype(np.float64), list(th.astype(np.float64))))
    ctx.close()


@pytest.mark.parametrize("nq", [16, 65])
@pytest.mark.parametrize("heads", [(1, 3), (4, 40)], ids=["small", "beyond"])
def test_recorded_decisions_at_the_edges(heads, nq):
    """The words a recording forward leaves, with about half of the decisions taken, so that a bit in the wrong place shows: the
    oracle's own decisions except within rounding of the threshold (the forward's error bar times the largest value of the row's
    layer); and the gradients from them (decisions handed to the oracle)."""
    B, H = heads
    T = 3
    w, inp, (Q, K, V), ctx = _setup(B, H, nq, 70, T, 0.3)
    phi = to_np(ctx.get_phi())
    binding.csat_set_i64(ctx.h, binding.CSAT_KEEP_MASKS, 1)
    G = wl.round_to_storage(np.random.default_rng(nq).standard_normal(inp["Q"].shape).astype(np.float32), "bf16")
    got = ctx.backward(Q, K, V, to_dev(G, "bf16"))
    words = ctx.backward_masks().cpu().numpy().astype(np.uint32)
    masks = np.stack([(words >> t) & 1 for t in range(T)], axis=2).astype(bool)
    kw = dict(T=T, lam=w.lam)
    stages = []
    orc.csat_backward(inp["Q"], inp["K"], inp["V"], phi, G, stages=stages, **kw)
    own = np.stack([s["masks"] for s in stages]).reshape(masks.shape)
    xs = np.abs(np.stack([s["xs"] for s in stages]).reshape(masks.shape))
    assert 0.3 <= own.mean() <= 0.7
    first = []
    orc.csat_forward(inp["Q"][:1], inp["K"][:1], inp["V"][:1], phi, T=1, lam=w.lam, stages=first)
    th = np.asarray([s["theta"] for s in first])[None, :, None, None, None]
    bar = TOL["bf16"] * xs.max(axis=(3, 4), keepdims=True)
    differ = masks != own
    assert (np.abs(xs - th)[differ] <= np.broadcast_to(bar, xs.shape)[differ]).all()
    assert differ.mean() <= 2e-2                            # entries within rounding of their threshold
    ref = orc.csat_backward(inp["Q"], inp["K"], inp["V"], phi, G, masks=masks, **kw)
    for nm, g, rf in zip(("dQ", "dK", "dV"), got, ref):
        assert rel_err(to_np(g), rf) <= TOL["bf16"], (heads, nq, nm, rel_err(to_np(g), rf))
    ctx.close()
