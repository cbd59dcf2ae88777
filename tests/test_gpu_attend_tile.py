"""bf16, d = 64: the kernel with one tile of 128 queries per CTA at its edges (queries around 32 and 128, measurements around
chunks of 64), on every side of the rules that choose its variants (two score buffers up to two tiles per SM, one beyond, B
folded into the values from eight on; one S_t, B_t per layer), against the float64 oracle within the parity bar.  (Of the first shape only
the per-layer check is this kernel's: the warp kernel serves the others.)"""
import numpy as np
import pytest
import torch

from oracle import csat_oracle as orc
from paper_2507_02957_b200 import binding, workloads as wl
from gpu_util import TOL, device_inputs, make_ctx, rel_err, to_dev, to_np

pytestmark = pytest.mark.gpu
D = 64


@pytest.mark.parametrize("B,H,nq,m", [(1, 50, 129, 64), (2, 70, 129, 64), (2, 70, 129, 67), (2, 48, 127, 65), (2, 80, 128, 131),
                                      (2, 120, 160, 193), (6, 60, 33, 200), (8, 152, 31, 70), (8, 152, 1, 129)])
def test_forward_at_the_edges(B, H, nq, m):
    T = 4
    w = wl.Workload("tile", B, H, 260, nq, D, m, "bf16", T, 0.001, "iid", 900 + nq)
    inp = wl.make_inputs(w)
    Q, K, V, _ = device_inputs(w, inp)
    ctx = make_ctx(w)
    phi = to_np(ctx.get_phi())
    r = np.random.default_rng(m)
    Psi = wl.round_to_storage((np.eye(D) + 0.3 * r.standard_normal((D, D)) / 8).astype(np.float32), "bf16")

    def check(**kw):
        ref = orc.csat_forward(inp["Q"], inp["K"], inp["V"], phi, **kw)
        out = to_np(ctx.forward(Q, K, V))
        assert np.isfinite(out).all() and np.abs(ref).max() > 0
        assert rel_err(out, ref) <= TOL["bf16"], (list(kw), rel_err(out, ref))

    for T in (1, 2, 4):
        ctx.set(T=T)
        check(T=T, lam=w.lam)
    ctx.set_dictionary(to_dev(Psi, "bf16"))
    check(T=4, lam=w.lam, Psi=Psi.astype(np.float64))
    S = wl.round_to_storage((0.6 * np.eye(D) + 0.4 * r.standard_normal((3, H, D, D)) / 8).astype(np.float32), "bf16")
    Bm = wl.round_to_storage((r.standard_normal((3, H, D, D)) / 8).astype(np.float32), "bf16")
    th = (0.02 * r.uniform(0.2, 1.5, size=(3, H))).astype(np.float32)
    ctx.set(T=3)
    ctx.set_lista_layer_weights(to_dev(S, "bf16"), to_dev(Bm, "bf16"), torch.from_numpy(th).cuda())
    check(T=3, lam=0.0, Psi=Psi.astype(np.float64), weights=(S.astype(np.float64), Bm.astype(np.float64), list(th.astype(np.float64))))
    ctx.close()


@pytest.mark.parametrize("nq,m", [(65, 64), (80, 131), (97, 65), (112, 200), (113, 64), (128, 64), (113, 65)])
def test_the_rule_between_this_kernel_and_128_queries_per_cta_of_the_warp_kernel(nq, m):
    """120 heads of up to 128 queries: eight warps of 16 queries up to 112 queries or with one chunk of measurements, this kernel
    otherwise; the plain and the recording forward."""
    w = wl.Workload("warp8", 2, 60, 230, nq, D, m, "bf16", 3, 0.001, "iid", 300 + nq)
    inp = wl.make_inputs(w)
    Q, K, V, _ = device_inputs(w, inp)
    ctx = make_ctx(w)
    phi = to_np(ctx.get_phi())
    ref = orc.csat_forward(inp["Q"], inp["K"], inp["V"], phi, T=3, lam=w.lam)
    for save in (0, 1):
        binding.csat_set_i64(ctx.h, binding.CSAT_SAVE_FOR_BACKWARD, save)
        out = to_np(ctx.forward(Q, K, V))
        assert np.isfinite(out).all() and rel_err(out, ref) <= TOL["bf16"], (save, rel_err(out, ref))
    ctx.close()
