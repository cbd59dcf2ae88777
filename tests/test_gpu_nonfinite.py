"""Values that are not finite: what a (batch, head) with a NaN or an infinity in its values leaves, beside heads that are finite."""
import pytest
import torch

from paper_2507_02957_b200 import binding

pytestmark = pytest.mark.gpu


def _randn(seed, *shape, dtype=torch.bfloat16):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda").to(dtype)


@pytest.mark.parametrize("d, H, n_q", [(64, 2, 70), (64, 40, 300), (128, 2, 70), (128, 3, 300)])
def test_decisions_of_rows_that_are_not_finite(d, H, n_q):
    """|NaN| > theta is false: a NaN in the values of head 0 makes every pre-activation of that head NaN, and none of its
    decisions is recorded as taken; the other heads' decisions and gradients keep their bits."""
    T, m = 5, 128
    ctx = binding.Csat(256, m, d, H, 3, n_q=n_q, dtype="bf16", T=T, lam=1e-3)
    binding.csat_set_i64(ctx.h, binding.CSAT_KEEP_MASKS, 1)
    Q, K, V, G = _randn(1, 1, H, n_q, d), _randn(2, 1, H, 256, d), _randn(3, 1, H, 256, d), _randn(4, 1, H, n_q, d)
    clean = [g.clone() for g in ctx.backward(Q, K, V, G)]
    words = ctx.backward_masks().clone()
    assert (words[0, 0] != 0).any()
    V[0, 0, 17, 5] = float("nan")
    dirty = ctx.backward(Q, K, V, G)
    got = ctx.backward_masks()
    assert (got[0, 0] == 0).all()
    assert torch.equal(got[:, 1:], words[:, 1:])
    for a, b in zip(dirty, clean):
        assert torch.equal(a[:, 1:], b[:, 1:])
    ctx.close()
