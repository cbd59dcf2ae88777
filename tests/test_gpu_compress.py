"""bf16 compression on the tensor cores, one shape or more for every way a measurement tile is dealt out (K and V columns together
or in CTAs of their own, one or two tiles per CTA, a batch element alone, a matrix of its own for the values), with ragged token and
measurement counts and an odd batch: K~ and V~ against float64 products with the matrix the library exports.

Bound: the result is rounded to bf16 once, 2^-8 of itself.  The products of bf16 numbers are exact in float32; the roundings of their sum
act like n random ones of 2^-24 of partial sums that grow to the result's typical size: sqrt(n) 2^-24 <= 2e-6 of the largest (n <= 1100),
and four times that is allowed (2e-3 2^-8 = 7.8e-6)."""
import numpy as np
import pytest
import torch

from paper_2507_02957_b200 import binding
from gpu_util import to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,n,m,d", [
    (3, 4, 331, 200, 64),       # d = 64, K and V apart, an odd batch
    (2, 16, 1000, 512, 64),     # the same with four tiles
    (9, 12, 333, 129, 64),      # one tile per CTA; the second tile has one row
    (5, 40, 200, 130, 64),      # two tiles per CTA
    (7, 20, 1100, 511, 64),     # the same, odd batch, ragged in everything
    (8, 30, 400, 300, 64),      # three tiles
    (1, 20, 700, 190, 64),      # a batch of one
    (2, 8, 777, 187, 128),      # d = 128, K and V apart
    (3, 25, 515, 135, 128),     # one tile per CTA, K and V together
    (4, 32, 300, 256, 128),     # two tiles per CTA
])
def test_compression_of_every_kind(B, H, n, m, d):
    ctx = binding.Csat(n, m, d, H, 3, B=B, n_q=16, dtype="bf16", T=1, lam=0.05)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + m)
    K, V = (torch.randn(B, H, n, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    Q = torch.randn(B, H, 16, d, generator=g, device="cuda").bfloat16()
    ctx.forward(Q, K, V)
    phi = torch.from_numpy(to_np(ctx.get_phi())).cuda()
    for got, x in zip(ctx.get_compressed(), (K, V)):
        ref = phi @ x.double()
        bound = 2.0 ** -8 * ref.abs() + 2e-3 * 2.0 ** -8 * ref.abs().max()
        assert got.shape == ref.shape and bool(((got.double() - ref).abs() <= bound).all()), (got.double() - ref).abs().max().item()
    ctx.close()


@pytest.mark.parametrize("B,H,n,m,d", [(3, 5, 331, 200, 64), (1, 9, 515, 129, 64), (2, 6, 777, 187, 128)])
def test_compression_with_a_matrix_of_its_own_for_the_values(B, H, n, m, d):
    ctx = binding.Csat(n, m, d, H, 3, B=B, n_q=16, dtype="bf16", T=1, lam=0.05)
    ctx.set(separate_phi=True)
    g = torch.Generator(device="cuda")
    g.manual_seed(n + m)
    K, V = (torch.randn(B, H, n, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    ctx.forward(torch.randn(B, H, 16, d, generator=g, device="cuda").bfloat16(), K, V)
    phi = torch.from_numpy(to_np(ctx.get_phi())).cuda()
    assert not torch.equal(phi[:H], phi[H:])
    for got, x, p in zip(ctx.get_compressed(), (K, V), (phi[:H], phi[H:])):
        ref = p @ x.double()
        bound = 2.0 ** -8 * ref.abs() + 2e-3 * 2.0 ** -8 * ref.abs().max()
        assert got.shape == ref.shape and bool(((got.double() - ref).abs() <= bound).all()), (got.double() - ref).abs().max().item()
    ctx.close()


@pytest.mark.parametrize("B,H,n,m,d", [
    (9, 12, 1500, 270, 64),     # one group of two parts of 144 measurements, an odd batch
    (16, 8, 1600, 392, 64),     # (tiles: too short)
    (16, 8, 2000, 392, 64),     # two parts of 208
    (5, 16, 2000, 600, 64),     # three groups of one part of 208
    (7, 10, 1030, 513, 64),     # the last group ends at its 161st row
    (2, 16, 2100, 300, 128),    # (tiles: one per SM, too few stages)
    (2, 12, 3001, 530, 128),    # (tiles)
    (1, 4, 4100, 3000, 128),    # sixteen groups of one part, K and V features in the two CTAs
])
def test_compression_on_pairs_of_ctas(B, H, n, m, d):
    """Features in M, measurements in N; the host-buffer forward compresses a head at a time on single CTAs: the same bits."""
    ctx = binding.Csat(n, m, d, H, 3, B=B, n_q=16, dtype="bf16", T=1, lam=0.05)
    g = torch.Generator(device="cuda").manual_seed(n + m)
    K, V = (torch.randn(B, H, n, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    Q = torch.randn(B, H, 16, d, generator=g, device="cuda").bfloat16()
    out = ctx.forward(Q, K, V)
    phi = torch.from_numpy(to_np(ctx.get_phi())).cuda()
    got = ctx.get_compressed()
    for y, x in zip(got, (K, V)):
        ref = phi @ x.double()
        bound = 2.0 ** -8 * ref.abs() + 8e-3 * 2.0 ** -8 * ref.abs().max()      # sqrt(n) twice that of the shapes above
        assert y.shape == ref.shape and bool(((y.double() - ref).abs() <= bound).all()), (y.double() - ref).abs().max().item()
    host = torch.empty(Q.shape, dtype=Q.dtype)
    ctx.forward_host(Q.cpu(), K.cpu(), V.cpu(), host)
    assert torch.equal(host, out.cpu()) and all(torch.equal(a, b) for a, b in zip(got, ctx.get_compressed()))
    ctx.close()


@pytest.mark.parametrize("B,H,n,m,d", [
    (32, 12, 197, 64, 64),      # one tile of measurements, a ragged token count
    (5, 30, 333, 65, 64),       # (90 tiles: one CTA per SM)
    (5, 60, 333, 65, 64),       # two batch elements per CTA, the last one alone; 180 tiles
    (1, 160, 500, 100, 64),     # a lone batch: K and V of one (batch, head) per tile
    (7, 16, 400, 140, 128),     # an odd batch
    (1, 160, 203, 128, 128),
    (5, 100, 260, 70, 64),      # 300 tiles: three rounds of one for two of two, a short token axis
    (2, 150, 1200, 128, 128),   # (a longer one: one CTA per SM)
])
def test_compression_with_two_ctas_per_sm(B, H, n, m, d):
    """More tiles than SMs; a head at a time (the host-buffer forward) has fewer, with one CTA per SM: the same bits."""
    ctx = binding.Csat(n, m, d, H, 3, B=B, n_q=16, dtype="bf16", T=1, lam=0.05)
    g = torch.Generator(device="cuda").manual_seed(n + m)
    K, V = (torch.randn(B, H, n, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    Q = torch.randn(B, H, 16, d, generator=g, device="cuda").bfloat16()
    out = ctx.forward(Q, K, V)
    phi = torch.from_numpy(to_np(ctx.get_phi())).cuda()
    got = ctx.get_compressed()
    for y, x in zip(got, (K, V)):
        ref = phi @ x.double()
        bound = 2.0 ** -8 * ref.abs() + 2e-3 * 2.0 ** -8 * ref.abs().max()
        assert y.shape == ref.shape and bool(((y.double() - ref).abs() <= bound).all()), (y.double() - ref).abs().max().item()
    host = torch.empty(Q.shape, dtype=Q.dtype)
    ctx.forward_host(Q.cpu(), K.cpu(), V.cpu(), host)
    assert torch.equal(host, out.cpu()) and all(torch.equal(a, b) for a, b in zip(got, ctx.get_compressed()))
    ctx.close()


@pytest.mark.parametrize("B,H,n,m,d", [
    (13, 4, 1517, 361, 128),    # one group of two parts
    (6, 8, 3000, 423, 128),     # three groups of one part, two CTAs per SM
    (2, 12, 3300, 927, 128),    # three groups of two parts
    (7, 16, 1600, 260, 128),    # more CTAs than SMs, one on each
    (11, 8, 2600, 441, 64),     # an odd batch, three groups of one part
])
def test_compression_on_pairs_of_ctas_where_it_is_chosen(B, H, n, m, d):
    test_compression_on_pairs_of_ctas(B, H, n, m, d)


@pytest.mark.parametrize("B,H,n,m,d,separate", [
    (3, 8, 636, 116, 32, False),       # the warp kernel: few tiles
    (6, 6, 1053, 111, 8, False),
    (2, 6, 700, 157, 56, False),
    (2, 5, 900, 150, 40, True),
    (3, 50, 140, 129, 32, False),      # the kernel of 64 columns: two batch elements per CTA, an odd batch
    (17, 24, 100, 40, 40, False),      # two CTAs per SM
    (5, 60, 130, 70, 48, False),
    (1, 16, 800, 540, 8, False),       # a lone batch
    (1, 160, 300, 100, 56, False),     # with two CTAs per SM
    (3, 50, 140, 129, 32, True),       # a matrix of their own for the values
    (1, 6, 300, 129, 72, False),       # the kernel of 128 columns: K and V apart
    (4, 32, 150, 100, 96, False),      # together
    (3, 60, 150, 120, 120, False),     # two CTAs per SM
    (2, 9, 333, 130, 88, True),
])
def test_compression_of_other_head_sizes(B, H, n, m, d, separate):
    """Both kernels that whole launches go to, either side of the choice between them."""
    ctx = binding.Csat(n, m, d, H, 3, B=B, n_q=16, dtype="bf16", T=0, lam=0.05)
    ctx.set(separate_phi=separate)
    g = torch.Generator(device="cuda").manual_seed(n + m)
    K, V = (torch.randn(B, H, n, d, generator=g, device="cuda").bfloat16() for _ in range(2))
    ctx.forward(torch.randn(B, H, 16, d, generator=g, device="cuda").bfloat16(), K, V)
    phi = torch.from_numpy(to_np(ctx.get_phi())).cuda()
    for got, x, p in zip(ctx.get_compressed(), (K, V), (phi[:H], phi[-H:])):
        ref = p @ x.double()
        bound = 2.0 ** -8 * ref.abs() + 2e-3 * 2.0 ** -8 * ref.abs().max()
        assert got.shape == ref.shape and bool(((got.double() - ref).abs() <= bound).all()), (got.double() - ref).abs().max().item()
    ctx.close()


@pytest.mark.parametrize("limit_us", [200, 3000])
def test_a_pair_of_ctas_gives_up_together(limit_us):
    """The functions that the kernels on pairs of CTAs end with after a wait that ran out: both CTAs' waits end (long before their own
    limit), and what only one of the producers had requested is complete when the pair ends.  998: it was not."""
    ctx = binding.Csat(64, 64, 64, 1, 3, dtype="bf16", T=1, lam=0.05)
    for _ in range(3):
        assert binding.csat_selftest_wait_timeout(ctx.h, limit_us) == 7
        assert "self-test" in binding.csat_last_error(ctx.h)
        assert binding.csat_clear_status(ctx.h) == 999
    ctx.close()
