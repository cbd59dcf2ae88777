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
    ctx.set(T=0)
    _check(ctx, Q, K, V, "no decoder", T=0, lam=0.0)
    ctx.set(T=T)
    S = (0.6 * torch.eye(D, device="cuda") + 0.05 * _randn(g, H, D, D)).bfloat16()
    Bm = (0.125 * _randn(g, H, D, D)).bfloat16()
    theta = 0.02 * (0.2 + 1.3 * torch.rand(T, H, generator=g, device="cuda"))
    for th in (theta, theta[:1]):
        ctx.set_lista_weights(S, Bm, th.contiguous())
        each = th.expand(T, H)
        _check(ctx, Q, K, V, ("weights", len(th)), T=T, lam=0.0,
               weights=lambda h: (to_np(S[h]), to_np(Bm[h]), [float(x) for x in each[:, h]]))
    for L in (1, T):                                            # one S_t, B_t per layer
        Sl, Bl = (x[None] + 0.02 * _randn(g, L, H, D, D) for x in (S.float(), Bm.float()))
        Sl, Bl = Sl.bfloat16(), Bl.bfloat16()
        ctx.set(T=L)
        ctx.set_lista_layer_weights(Sl, Bl, theta[:L].contiguous())
        _check(ctx, Q, K, V, ("layers", L), T=L, lam=0.0,
               weights=lambda h: (to_np(Sl[:, h]), to_np(Bl[:, h]), [float(x) for x in theta[:L, h]]))
    ctx.close()


@pytest.mark.parametrize("B,H,nq,m", [
    (1, 12, 100, 200),      # 64 queries per CTA of the warp kernel
    (2, 50, 90, 190),       # 128
    (2, 80, 128, 250),      # two score buffers
    (2, 140, 250, 200),
    (2, 120, 160, 200),     # one
    (8, 152, 31, 200),      # B folded into the values
])
def test_scores_that_rise_from_chunk_to_chunk(B, H, nq, m):
    """Row r of K~ is near u r / 64: a row's scores rise (or fall, by the sign of its query) by about 7 = 10 log2 units a chunk of 64, more
    than the 8 that a reference may lag behind, so that every chunk rescales what half of a warp's rows have summed up.  K~ is rounded to
    2^-9 of its values, which moves a score of at most 36 by 36 2^-9 / sqrt(64) = 0.9 %."""
    n, T, lam = 256, 3, 1e-3
    g = torch.Generator(device="cuda").manual_seed(m)
    u = (2 * torch.randint(0, 2, (D,), generator=g, device="cuda") - 1).float()
    sign = (2 * torch.randint(0, 2, (B, H, nq, 1), generator=g, device="cuda") - 1).float()
    Q = (sign * u + 0.1 * _randn(g, B, H, nq, D)).bfloat16()
    K = (u + 0.2 * _randn(g, B, H, n, D)).bfloat16()
    V = _randn(g, B, H, n, D).bfloat16()
    ramp = 0.875 * torch.arange(m, device="cuda") / 64 / n
    phi = (ramp[None, :, None] + 0.04 / n ** 0.5 * _randn(g, H, m, n)).bfloat16()
    ctx = binding.Csat(n, m, D, H, 3, B=B, n_q=nq, dtype="bf16", T=T, lam=lam)
    ctx.set_phi(phi)
    st = {}
    orc.csat_forward_head(to_np(Q[0, 0]), to_np(K[0, 0]), to_np(V[0, 0]), to_np(phi[0]), T=0, lam=0.0, stages=st)
    s = np.sign(to_np(sign[0, 0])) * (to_np(Q[0, 0]) @ st["Kt"].T) / 8 / np.log(2)
    tops = [s[:, c:c + 64].max(1) for c in range(0, m - m % 64, 64)]
    assert all((b - a > 8).mean() > 0.8 for a, b in zip(tops, tops[1:]))
    eye = (torch.eye(D, device="cuda") + 0.03 * _randn(g, H, D, D)).bfloat16()
    ctx.set(T=0)
    _check(ctx, Q, K, V, "no decoder", T=0, lam=0.0)
    ctx.set(T=T)
    ctx.set_decoder_matrix(eye)
    _check(ctx, Q, K, V, "derived", T=T, lam=lam, D=lambda h: to_np(eye[h]))
    th = torch.full((T, H), 1e-3, device="cuda")
    Sl, Bl = (x[None].expand(T, H, D, D).contiguous() for x in (0.1 * eye, eye))
    ctx.set_lista_layer_weights(Sl, Bl, th)
    _check(ctx, Q, K, V, "per layer", T=T, lam=0.0, weights=lambda h: (to_np(Sl[:, h]), to_np(Bl[:, h]), [1e-3] * T))
    ctx.close()
