"""bf16, d = 64: what the two attention / recovery kernels do where it depends on the size of the job (148 SMs): score buffers and chunks in
flight, one or several thresholds, and the accumulator's rescaling when scores rise.  Sampled (batch, head) pairs against the float64
oracle within the parity bar."""
import numpy as np
import pytest
import torch

from oracle import csat_oracle as orc
from paper_2507_02957_b200 import binding
from gpu_util import TOL, rel_err, to_np

pytestmark = pytest.mark.gpu
D = 64


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _check(ctx, Q, K, V, what, **kw):
    """The plain and the recording forward."""
    B, H = Q.shape[:2]
    phi = ctx.get_phi()
    for save in (0, 1):
        binding.csat_set_i64(ctx.h, binding.CSAT_SAVE_FOR_BACKWARD, save)
        out = ctx.forward(Q, K, V)
        assert torch.isfinite(out).all() and torch.equal(out, ctx.forward(Q, K, V)), what
        for b, h in ((0, 0), (B // 2, H // 2), (B - 1, H - 1)):
            args = {k: v(h) if callable(v) else v for k, v in kw.items()}
            ref = orc.csat_forward_head(*(to_np(x[b, h]) for x in (Q, K, V)), to_np(phi[h]), **args)
            err = rel_err(to_np(out[b, h]), ref)
            assert np.abs(ref).max() > 0 and err <= TOL["bf16"], (what, save, b, h, err)
    binding.csat_set_i64(ctx.h, binding.CSAT_SAVE_FOR_BACKWARD, 0)


@pytest.mark.parametrize("B,H,nq,m", [
    (2, 64, 77, 192),       # 128 queries per CTA of the warp kernel, up to three chunks
    (2, 64, 77, 193),       # two score buffers, four chunks in flight
    (1, 60, 150, 257),
    (1, 60, 150, 520),
    (2, 70, 129, 64),       # 280 tiles, the second of a head has one row
    (2, 70, 129, 131),
    (2, 99, 150, 64),       # 396 tiles: one buffer
    (2, 140, 250, 64),      # 560: one buffer for a single chunk
    (2, 140, 250, 131),     # two for more
    (2, 149, 250, 131),     # 596: one
])
def test_thresholds_and_sizes(B, H, nq, m):
    n, T = 530, 4
    g = torch.Generator(device="cuda").manual_seed(nq + m)
    Q, K, V = (_randn(g, B, H, r, D).bfloat16() for r in (nq, n, n))
    ctx = binding.Csat(n, m, D, H, 3, B=B, n_q=nq, dtype="bf16", T=T, lam=0.001)
    _check(ctx, Q, K, V, "one threshold", T=T, lam=0.001)
    ctx.set(lam=0.0)
    _check(ctx, Q, K, V, "no threshold", T=T, lam=0.0)
    S = (0.6 * torch.eye(D, device="cuda") + 0.05 * _randn(g, H, D, D)).bfloat16()
    Bm = (0.125 * _randn(g, H, D, D)).bfloat16()
    theta = 0.02 * (0.2 + 1.3 * torch.rand(T, H, generator=g, device="cuda"))
    for th in (theta, theta[:1]):
        ctx.set_lista_weights(S, Bm, th.contiguous())
        each = th.expand(T, H)
        _check(ctx, Q, K, V, ("weights", len(th)), T=T, lam=0.0,
               weights=lambda h: (to_np(S[h]), to_np(Bm[h]), [float(x) for x in each[:, h]]))
    ctx.close()
