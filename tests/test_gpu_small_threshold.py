"""bf16: thresholds mu lambda that are zero, below the normal numbers or barely above in float32.  The kernels that run the recurrence in
units of 2 theta take such thresholds in the data's units; the float64 oracle within the parity bar, one shape for each kernel and
variant the plain forward chooses."""
import numpy as np
import pytest

from oracle import csat_oracle as orc
from paper_2507_02957_b200 import workloads as wl
from gpu_util import TOL, device_inputs, make_ctx, rel_err, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,nq,d,m", [
    (1, 6, 100, 64, 64),        # 64 queries per CTA of the warp kernel
    (2, 60, 100, 64, 64),       # 128
    (2, 80, 128, 64, 131),      # one tile per CTA, two score buffers
    (2, 120, 160, 64, 70),      # one score buffer
    (8, 152, 31, 64, 70),       # B folded into the values
    (1, 6, 300, 128, 130),      # two tiles per CTA
    (2, 80, 130, 128, 130),     # the same, folded
])
def test_threshold_at_the_bottom_of_float32(B, H, nq, d, m):
    T = 4
    w = wl.Workload("small_theta", B, H, 260, nq, d, m, "bf16", T, 0.001, "iid", 700 + nq)
    inp = wl.make_inputs(w)
    Q, K, V, _ = device_inputs(w, inp)
    ctx = make_ctx(w)
    phi = to_np(ctx.get_phi())
    for lam in (1e-60, 1e-40, 1e-38, 1e-22, 1e-12):
        ctx.set(lam=lam)
        out = to_np(ctx.forward(Q, K, V))
        ref = orc.csat_forward(inp["Q"], inp["K"], inp["V"], phi, T=T, lam=lam)
        assert np.isfinite(out).all() and np.abs(ref).max() > 0, lam
        assert rel_err(out, ref) <= TOL["bf16"], (lam, rel_err(out, ref))
    ctx.close()
