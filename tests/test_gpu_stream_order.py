"""`csat_attend` directly behind a kernel of the library that may still be running: one that writes its queries (the input
projection, another attention), or one that writes its decoder (the set-up after a changed parameter).  Attention kernels may start before the kernel in front has finished; every result has to
have the bits of the same call made after a synchronisation.  A buffer that could be read too early holds other finite values
before the calls."""
import pytest
import torch

from paper_2507_02957_b200 import binding

pytestmark = pytest.mark.gpu


def _randn(seed, *shape, dtype=torch.bfloat16):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda").to(dtype)


def _context(d, H, n, T, seed=5, dtype="bf16", lam=1e-3):
    """A context whose K~|V~ are those of random keys and values."""
    ctx = binding.Csat(n, 128, d, H, seed, dtype=dtype, T=T, lam=lam)
    ctx.forward(*(_randn(seed + i, 1, H, n, d, dtype=ctx.torch_dtype) for i in range(3)))
    torch.cuda.synchronize()
    return ctx


# heads, tokens: a few tiles (at d = 64 the warp-level kernel's), more than one CTA of 64 queries per SM, about a wave of pairs of
# 128 queries; none long enough for B to be folded into the values by a kernel in between
SIZES = [(4, 1024), (6, 1600), (16, 2304)]
sizes = pytest.mark.parametrize("d, T, H, n", [(d, T, *s) for d in (64, 128) for T in (0, 10) for s in SIZES])


def _check(calls, buffers, others):
    """`calls` (back to back) writes `buffers`; the same with a synchronisation after each gives the bits to compare with."""
    for f in calls:
        f()
        torch.cuda.synchronize()
    want = [b.clone() for b in buffers]
    for _ in range(5):
        for b, o in zip(buffers, others):
            b.copy_(o)
        torch.cuda.synchronize()
        for f in calls:
            f()
        torch.cuda.synchronize()
        for b, w in zip(buffers, want):
            assert torch.equal(b, w)


@sizes
def test_attend_behind_the_projection(d, T, H, n):
    ctx = _context(d, H, n, T)
    dm = 512
    X, W = _randn(11, 1, n, dm), _randn(12, dm, 3 * H * d) * dm ** -0.5
    Q, K, V, out = (torch.empty(1, H, n, d, dtype=torch.bfloat16, device="cuda") for _ in range(4))
    _check([lambda: binding.csat_project_qkv(ctx.h, X, X, W, dm, Q, K, V), lambda: ctx.attend(Q, out=out)],
           [Q, out], [_randn(13, *Q.shape), _randn(14, *Q.shape)])
    ctx.close()


@sizes
def test_attend_behind_attend_and_forward(d, T, H, n):
    """attend(attend(Q)) on one memory, and attend on another context's forward."""
    first, second = _context(d, H, n, T), _context(d, H, n, T, seed=25)
    Q = _randn(21, 1, H, n, d)
    mid, out = torch.empty_like(Q), torch.empty_like(Q)
    others = [_randn(22, *Q.shape), _randn(23, *Q.shape)]
    _check([lambda: first.attend(Q, out=mid), lambda: first.attend(mid, out=out)], [mid, out], others)
    K, V = _randn(24, *Q.shape), _randn(25, *Q.shape)
    _check([lambda: first.forward(Q, K, V, out=mid), lambda: second.attend(mid, out=out)], [mid, out], others)
    first.close()
    second.close()


@pytest.mark.parametrize("weights", ["derived", "supplied", "per_layer"])
@pytest.mark.parametrize("dtype, d, H, n", [("bf16", 64, 4, 1024), ("bf16", 64, 6, 1600), ("bf16", 128, 6, 1600), ("bf16", 96, 2, 300),
                                            ("fp32", 64, 1, 300), ("fp32", 128, 1, 300)])
def test_attend_behind_the_decoder_set_up(dtype, d, H, n, weights):
    """A changed step size (S, B and the threshold depend on it), or other supplied weights, and at once an attention."""
    ctx = _context(d, H, n, 10, dtype=dtype)
    dt = ctx.torch_dtype
    Q = _randn(31, 1, H, n, d, dtype=dt)
    out = torch.empty_like(Q)
    eye = torch.eye(d, device="cuda")
    S = [(0.6 * eye + 0.3 * d ** -0.5 * _randn(40 + i, H, d, d, dtype=torch.float32)).to(dt) for i in (0, 1)]
    Bm = [(_randn(50 + i, H, d, d, dtype=torch.float32) * d ** -0.5).to(dt) for i in (0, 1)]
    th = [torch.full((1, H), x, device="cuda") for x in (0.01, 0.03)]

    def change(i):
        if weights == "per_layer":
            ctx.set_lista_layer_weights(S[i].expand(10, H, d, d).contiguous(), Bm[i].expand(10, H, d, d).contiguous(),
                                        th[i].expand(10, H).contiguous())
        elif weights == "supplied":
            ctx.set_lista_weights(S[i], Bm[i], th[i])
        else:
            ctx.set(step=(0.05, 0.1)[i])

    want = []
    for i in (0, 1):
        change(i)
        ctx.get_decoder()
        torch.cuda.synchronize()
        want.append(ctx.attend(Q).clone())
        torch.cuda.synchronize()
    assert not torch.equal(*want)
    for k in range(10):
        change(k % 2)
        ctx.attend(Q, out=out)
        torch.cuda.synchronize()
        assert torch.equal(out, want[k % 2])
    ctx.close()
