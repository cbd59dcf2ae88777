"""Values that are not finite: what a (batch, head) with a NaN or an infinity in its values leaves, beside heads that are finite."""
import pytest
import torch

from paper_2507_02957_b200 import binding

pytestmark = pytest.mark.gpu


def _randn(seed, *shape, dtype=torch.bfloat16):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda").to(dtype)


@pytest.mark.parametrize("d, H, n_q", [(64, 2, 70), (64, 40, 300), (64, 110, 300), (128, 2, 70), (128, 3, 300)])
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


def _infinite_head(d, H, n_q, m, T, dtype, sign):
    """Positive measurements and decoder matrices, and one infinity in the values of head 0: every sum of that head that meets
    it is an infinity of its sign, no two of different signs meet."""
    ctx = binding.Csat(200, m, d, H, 3, n_q=n_q, dtype=dtype, T=T, lam=1e-3)
    dt = ctx.torch_dtype
    ctx.set_phi((0.1 + _randn(1, H, m, 200, dtype=torch.float32).abs()).to(dt))
    if T > 0:
        S, Bm = ((0.01 + _randn(i, H, d, d, dtype=torch.float32).abs() / d).to(dt) for i in (2, 3))
        ctx.set_lista_weights(S, Bm, torch.full((1, H), 0.01, device="cuda"))
    Q, K, V = (0.05 * _randn(10 + i, 1, H, n, d, dtype=torch.float32) for i, n in enumerate((n_q, 200, 200)))
    Q, K, V = Q.to(dt), K.to(dt), V.to(dt)
    V2 = V.clone()
    V2[0, 0, 17, 5] = sign * float("inf")
    return ctx, Q, K, V, V2


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("T", [0, 1, 4])
@pytest.mark.parametrize("d", [8, 24, 40, 64, 72, 96, 120, 128])
def test_infinities_in_float32(d, T, sign):
    """An infinity stays one through the float32 kernels, padded head sizes included, and is a decision in every layer."""
    H, n_q = 2, 70
    ctx, Q, K, V, V2 = _infinite_head(d, H, n_q, 50, T, "fp32", sign)
    want = ctx.forward(Q, K, V).clone()
    got = ctx.forward(Q, K, V2)
    assert torch.isfinite(want).all() and torch.equal(got[:, 1:], want[:, 1:])
    if T == 0:
        assert (got[0, 0, :, 5] == sign * float("inf")).all()
        got[0, 0, :, 5], want[0, 0, :, 5] = 0, 0
        assert torch.equal(got, want)
    else:
        assert (got[0, 0] == sign * float("inf")).all()
        binding.csat_set_i64(ctx.h, binding.CSAT_KEEP_MASKS, 1)
        ctx.backward(Q, K, V2, _randn(4, 1, H, n_q, d, dtype=torch.float32))
        assert (ctx.backward_masks()[0, 0] == (1 << T) - 1).all()
    ctx.close()


@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("T", [0, 1, 4])
@pytest.mark.parametrize("d", [8, 24, 40, 72, 96, 120])
def test_infinities_in_two_bf16_parts(d, T, sign):
    """The same for bf16 storage at head sizes whose float32 values go through the matrix instructions in two parts (the second
    part of an infinity is NaN)."""
    H, n_q = 2, 70
    ctx, Q, K, V, V2 = _infinite_head(d, H, n_q, 50, T, "bf16", sign)
    want = ctx.forward(Q, K, V).clone()
    got = ctx.forward(Q, K, V2)
    assert torch.isfinite(want).all() and torch.equal(got[:, 1:], want[:, 1:])
    if T == 0:
        assert (got[0, 0, :, 5] == sign * float("inf")).all()
        got[0, 0, :, 5], want[0, 0, :, 5] = 0, 0
        # float32 throughout against two parts, rounded to bf16: at most one step (2^-7 of the value) apart
        assert ((got - want).abs() <= 2 ** -7 * want.abs()).all()
    else:
        assert (got[0, 0] == sign * float("inf")).all()
    ctx.close()


@pytest.mark.parametrize("d", [8, 40, 96, 120])
def test_where_two_bf16_parts_give_nan_and_infinity(d):
    """NaN and infinities of either sign in queries, keys and values: each output is finite, NaN or an infinity where the float32
    kernels' is (a few rows only: the rest of a head keeps what it had)."""
    H, n_q, n, m, T = 4, 70, 200, 130, 3
    ctx = binding.Csat(n, m, d, H, 3, n_q=n_q, dtype="bf16", T=T, lam=1e-3)
    Q, K, V = _randn(1, 1, H, n_q, d), _randn(2, 1, H, n, d), _randn(3, 1, H, n, d)
    Q[0, 0, 33, 1], Q[0, 0, 17, 2], Q[0, 0, 69, 0] = float("nan"), float("inf"), float("-inf")
    V[0, 1, 5, 3], K[0, 2, 199, d - 1] = float("-inf"), float("inf")
    for T in (0, 1, 3):
        ctx.set(T=T, force_simt=0)
        a = ctx.forward(Q, K, V).clone()
        ctx.set(force_simt=1)
        b = ctx.forward(Q, K, V)
        assert torch.equal(torch.isnan(a), torch.isnan(b)) and torch.equal(torch.isposinf(a), torch.isposinf(b))
        assert torch.equal(torch.isneginf(a), torch.isneginf(b))
        assert torch.isnan(a[0, 0, 33]).all() and torch.isfinite(a[0, 0, :17]).all() and torch.isfinite(a[0, 3]).all()
    ctx.close()
