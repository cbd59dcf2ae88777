"""bf16 contexts with head sizes that are no multiple of 64 on the tensor cores (one tile of 128 queries per CTA): edges of tiles, chunks of
measurements and padded heads, against float64 products of the library's own K~, V~ and decoder.

Bound: the output is rounded to bf16 once, 2^-8 of itself.  P, z and the iterates enter products in 16 bits (2^-16 each, in at most T + 2
products of a recurrence that does not grow), ex2 and the normalisation are good to 2^-21: together less than (T + 4) 2^-15 of the row's largest
value before the last shrinkage, which max |z B| stands for; three times that is allowed."""
import math

import pytest
import torch

from paper_2507_02957_b200 import binding

pytestmark = pytest.mark.gpu

#     B  H   n    n_q  m    d   T
SHAPES = [(2, 75, 70, 129, 64, 8, 3),
          (1, 150, 80, 128, 63, 24, 10),
          (3, 50, 140, 130, 129, 32, 12),
          (2, 80, 60, 1, 33, 16, 0),
          (1, 80, 150, 37, 65, 40, 1),
          (2, 40, 130, 127, 130, 56, 2),
          (1, 1, 100, 1, 72, 72, 7),
          (2, 3, 300, 257, 200, 80, 20),
          (1, 2, 97, 33, 96, 96, 2),
          (5, 33, 110, 129, 97, 96, 5)]


@pytest.mark.parametrize("B,H,n,nq,m,d,T", SHAPES)
@pytest.mark.parametrize("variant", ["derived", "no_threshold", "psi_thresholds_per_layer"])
def test_tile_kernel_against_float64(B, H, n, nq, m, d, T, variant):
    if variant != "derived" and T == 0:
        pytest.skip("no decoder without recovery layers")
    g = torch.Generator(device="cuda").manual_seed(n + d)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    Q, K, V = rnd(B, H, nq, d).bfloat16(), rnd(B, H, n, d).bfloat16(), rnd(B, H, n, d).bfloat16()
    ctx = binding.Csat(n, m, d, H, 3, B=B, n_q=nq, dtype="bf16", T=T, lam=0.0 if variant == "no_threshold" else 0.05)
    psi = torch.eye(d, dtype=torch.float64, device="cuda")
    if variant == "psi_thresholds_per_layer":
        psi = torch.linalg.qr(rnd(d, d))[0].bfloat16()
        ctx.set_dictionary(psi)
        S = (0.5 * torch.eye(d, device="cuda") + 0.3 * rnd(H, d, d) / math.sqrt(d)).bfloat16()
        thetas = 0.2 * torch.rand(T, H, generator=g, device="cuda")
        ctx.set_lista_weights(S, (rnd(H, d, d) / math.sqrt(d)).bfloat16(), thetas)
    elif m < d or n < d:
        pytest.skip("no derived decoder")
    out = ctx.forward(Q, K, V).double()
    assert torch.equal(out, ctx.forward(Q, K, V).double())
    Kt, Vt = (x.double() for x in ctx.get_compressed())
    z = torch.softmax(Q.double() @ Kt.transpose(-1, -2) / math.sqrt(d), -1) @ Vt
    ref, big = z, z.abs().amax(-1, keepdim=True)
    if T > 0:
        S, Bm, theta, _ = (x.double() for x in ctx.get_decoder())
        theta = thetas.double() if variant == "psi_thresholds_per_layer" else theta.expand(T, H)
        c = z @ Bm
        ref = torch.zeros_like(z)
        big = c.abs().amax(-1, keepdim=True)
        for t in range(T):
            th = theta[t].view(1, H, 1, 1)
            x = c + ref @ S
            ref = x - torch.minimum(torch.maximum(x, -th), th)
            big = torch.maximum(big, x.abs().amax(-1, keepdim=True))
        ref = ref @ psi.double().T
        big = big * math.sqrt(d) if variant == "psi_thresholds_per_layer" else big
    bound = 2.0 ** -8 * ref.abs() + 3 * (T + 4) * 2.0 ** -15 * big
    assert bool(((out - ref).abs() <= bound).all()), ((out - ref).abs() / bound).max().item()
    ctx.close()


@pytest.mark.parametrize("B,H,n,nq,m,d,T", [(1, 300, 80, 128, 63, 24, 10), (1, 150, 80, 128, 63, 24, 6), (2, 160, 40, 128, 40, 16, 5), (1, 152, 30, 127, 20, 8, 3)])
def test_tile_kernel_of_small_heads(B, H, n, nq, m, d, T):
    """Jobs at the ends of the choice: the tile kernel's."""
    test_tile_kernel_against_float64(B, H, n, nq, m, d, T, "psi_thresholds_per_layer")
