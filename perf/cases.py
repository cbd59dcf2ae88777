"""The work that users of this framework have it do, as cases that can be prepared, run and compared.

A case is a plain dict.  `pass` says which public entry points it takes:

  forward   `Csat.forward` on inputs that are in device memory
  layer     `Csat.project_qkv` (the input projections in front of the path), then `Csat.forward`
  train     `csat_attention` under torch.autograd and the gradients of Q, K, V
  learned   one step of a trained decoder: the step's measurement matrix and per-layer weights are set, forward,
            backward, and the gradients of the inputs, the layers' weights and the measurement matrix (the thresholds
            are not trained here)

Sizes are those of the workloads in `paper_2507_02957_b200/workloads.py` (197 tokens of an image, 196 patches a video
frame, 77 text tokens, sequences to 16384) or generic ones of the same kind.

The gradients are discontinuous where an iterate passes its threshold: there two correct implementations decide
differently and the gradients they give are percents apart (4 to 9 % at lambda = 0.05, between bf16 and float32 kernels of
this repository as between inputs a quarter of a bf16 step apart).  The training cases therefore have thresholds so low
that hardly an iterate lies near one, and queries scaled for scores of unit variance, so that no few rows carry dQ.
"""
import math

import torch

from paper_2507_02957_b200 import binding
from paper_2507_02957_b200.autograd import csat_attention

PATCHES = 196       # of an image or a video frame


def _case(name, kind, dtype, B, H, n, d, m, T, lam, *, n_q=None, data="iid", psi=False):
    c = {"pass": kind, "dtype": dtype, "B": B, "H": H, "n": n, "n_q": n if n_q is None else n_q, "d": d, "m": m, "T": T,
         "lam": lam, "data": data, "psi": psi}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call there is: one head, 256 tokens, in float32 (a latency, not a throughput)
        _case("tiny_fp32", "forward", "fp32", 1, 1, 256, 64, 64, 10, 0.1),
        # serving one image: 12 heads over 196 patches and a class token
        _case("image_one", "forward", "bf16", 1, 12, 197, 64, 64, 10, 0.1),
        # an attention layer over a batch of 32 such images, from the layer's tokens (768 = 12 x 64 features) on
        _case("image_layer", "layer", "bf16", 32, 12, 197, 64, 64, 10, 0.1),
        # self-attention over 8-frame clips, whose frames repeat each other
        _case("video", "forward", "bf16", 8, 12, 1568, 64, 256, 20, 0.05, data="video"),
        # 77 text queries over 16-frame clips, values sparse in a dictionary (few queries: the decode-like direction)
        _case("text_to_video", "forward", "bf16", 16, 8, 3136, 64, 392, 20, 0.05, n_q=77, data="video", psi=True),
        # a sequence of an odd length in the middle of the range, large heads
        _case("ragged", "forward", "bf16", 2, 16, 3001, 128, 187, 20, 0.05),
        # the longest sequences
        _case("long", "forward", "bf16", 2, 16, 16384, 128, 1024, 20, 0.05),
        # training on the video clips, decoder derived from Phi
        _case("video_train", "train", "bf16", 8, 12, 1568, 64, 256, 20, 1e-7, data="video"),
        # training on long sequences, large heads
        _case("long_train", "train", "bf16", 1, 16, 8192, 128, 512, 20, 1e-7),
        # training the decoder's layers and the measurement matrix themselves
        _case("learned_train", "learned", "bf16", 4, 12, 1568, 64, 256, 10, 1e-7, data="video"),
        # training in float32 at a size where that is affordable
        _case("fp32_train", "train", "fp32", 2, 8, 512, 64, 96, 10, 1e-7),
        # a head size between the usual two, which the general kernels serve
        _case("other_head_size", "forward", "bf16", 4, 8, 1024, 96, 128, 10, 0.05),
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# what draw() takes its sizes from: (weight, pass, dtype, head sizes, range of n, most flops: the listed case's)
_RANGES = [
    (5, "forward", "bf16", (64, 128), (128, 16384), "long"),
    (2, "layer", "bf16", (64, 128), (128, 2048), "image_layer"),
    (3, "train", "bf16", (64, 128), (128, 8192), "long_train"),
    (2, "learned", "bf16", (64, 128), (196, 1568), "learned_train"),
    (2, "forward", "fp32", (32, 64, 96, 128), (128, 2048), "fp32_train"),
    (2, "train", "fp32", (32, 64, 96), (128, 512), "fp32_train"),
    (1, "forward", "bf16", (32, 80, 96), (128, 1024), "other_head_size"),
]


def draw(rng):
    _, kind, dtype, heads, (lo, hi), most = rng.choices(_RANGES, weights=[r[0] for r in _RANGES])[0]
    most = work(next(c for c in listed() if c["name"] == most))["flops"]
    while True:
        d = rng.choice(heads)
        n = _log_between(rng, max(lo, d), hi)
        m = min(n, max(d, int(n / rng.uniform(3, 16))))
        T = rng.choice((5, 10, 20))
        n_q = rng.choice((n, n, _log_between(rng, 16, max(17, n)))) if kind == "forward" else n
        video = kind != "layer" and rng.random() < 0.4
        H = rng.choice((1, 4, 6, 8, 12, 16))
        lam = rng.choice((1e-7, 2e-7) if kind in ("train", "learned") else (0.02, 0.05, 0.1))
        c = _case(None, kind, dtype, 1, H, n, d, m, T, lam, n_q=n_q,
                  data="video" if video else "iid", psi=video and kind == "forward" and rng.random() < 0.5)
        room = int(most / work(c)["flops"])
        if room >= 1:
            return dict(c, B=_log_between(rng, 1, min(room, 48)))


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _tokens(case, g):
    """Rows of keys or values [B, H, n, d]: independent, or frames that repeat a base of 196 patches with noise."""
    B, H, n, d = (case[k] for k in ("B", "H", "n", "d"))
    if case["data"] != "video":
        return torch.randn(B, H, n, d, generator=g, device="cuda")
    base = torch.randn(B, H, PATCHES, d, generator=g, device="cuda")
    frames = -(-n // PATCHES)
    return base.repeat(1, 1, frames, 1)[:, :, :n] + 0.1 * torch.randn(B, H, n, d, generator=g, device="cuda")


def _inputs(case, seed):
    """Everything random about a case's state, drawn in one order for prepare() and exact()."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    dt = _dtype(case)
    B, H, n, n_q, d, m, T = (case[k] for k in ("B", "H", "n", "n_q", "d", "m", "T"))
    s = {}
    if case["pass"] == "layer":
        dm = H * d
        s["X"] = torch.randn(B, n, dm, generator=g, device="cuda").to(dt)
        s["W"] = (torch.randn(dm, 3 * dm, generator=g, device="cuda") / math.sqrt(dm)).to(dt)
        return s
    s["Q"] = torch.randn(B, H, n_q, d, generator=g, device="cuda").to(dt)
    s["K"] = _tokens(case, g).to(dt)
    if case["psi"]:
        # values that are sparse (a quarter of the coefficients) in an orthonormal dictionary
        psi = torch.linalg.qr(torch.randn(d, d, generator=g, device="cuda"))[0]
        keys = torch.rand(B, H, n, d, generator=g, device="cuda")
        beta = torch.randn(B, H, n, d, generator=g, device="cuda")
        beta *= keys < 0.25
        s["V"] = (beta @ psi.t()).to(dt)
        s["psi"] = psi.to(dt)
    else:
        s["V"] = _tokens(case, g).to(dt)
    if case["pass"] in ("train", "learned"):
        s["Q"] *= math.sqrt(m / n)          # rows of K~ = Phi K are sqrt(n / m) times as long as those of K
        s["dOut"] = torch.randn(B, H, n_q, d, generator=g, device="cuda").to(dt)
    if case["pass"] == "learned":
        # weights some way into training: the derived ones, moved a little, each layer by itself
        moved = 0.02 / math.sqrt(d)
        s["dS"] = moved * torch.randn(T, H, d, d, generator=g, device="cuda")
        s["dBm"] = moved * torch.randn(T, H, d, d, generator=g, device="cuda")
        s["dtheta"] = 0.5 + torch.rand(T, H, generator=g, device="cuda")
        s["phi"] = (torch.randn(H, m, n, generator=g, device="cuda") / math.sqrt(m)).to(dt)
    return s


def prepare(case, seed):
    B, H, n, n_q, d, m, T = (case[k] for k in ("B", "H", "n", "n_q", "d", "m", "T"))
    ctx = binding.Csat(n, m, d, H, 0, B=B, n_q=n_q, dtype=case["dtype"], T=T, lam=case["lam"])
    s = dict(_inputs(case, seed), case=case, ctx=ctx)
    if case["psi"]:
        ctx.set_dictionary(s["psi"])
    if case["pass"] in ("train", "learned"):
        for k in "QKV":
            s[k].requires_grad_(True)
    if case["pass"] == "learned":
        binding.csat_set_i64(ctx.h, binding.CSAT_WEIGHT_GRADS, 1)
        S, Bm, theta, _ = ctx.get_decoder()
        s["S"] = (S + s.pop("dS")).to(_dtype(case))
        s["Bm"] = (Bm + s.pop("dBm")).to(_dtype(case))
        s["theta"] = theta * s.pop("dtheta")
    return s


def run(state):
    ctx, kind = state["ctx"], state["case"]["pass"]
    if kind == "forward":
        return ctx.forward(state["Q"], state["K"], state["V"])
    if kind == "layer":
        Q, K, V = ctx.project_qkv(state["X"], state["W"])
        return ctx.forward(Q, K, V)
    Q, K, V = state["Q"], state["K"], state["V"]
    if kind == "learned":
        ctx.set_phi(state["phi"])
        ctx.set_lista_layer_weights(state["S"], state["Bm"], state["theta"])
    out = csat_attention(ctx, Q, K, V)
    grads = torch.autograd.grad(out, (Q, K, V), state["dOut"])
    if kind == "train":
        return (out.detach(),) + grads
    dS, dB, _, _ = ctx.weight_grads()
    return (out.detach(),) + grads + (dS, dB, ctx.backward_phi(K.detach(), V.detach()))


def work(case):
    B, H, n, n_q, d, m, T = (case[k] for k in ("B", "H", "n", "n_q", "d", "m", "T"))
    es = 2 if case["dtype"] == "bf16" else 4
    bh, kind = B * H, case["pass"]
    q, kv, phi = bh * n_q * d, bh * n * d, H * m * n            # elements of Q or out, of K or V, of Phi
    layer = 2 * bh * n_q * d * d                                # one product of the recurrence over all queries
    compress, attend = 4 * bh * m * n * d, 4 * bh * n_q * m * d
    flops = compress + attend + layer * (T + (1 if case["psi"] else 0))
    size = 2 * q + 2 * kv + phi                                 # elements in and out
    extra = 0                                                   # bytes of other types
    if kind == "layer":
        dm = H * d
        flops += 2 * B * n * dm * 3 * dm
        size = B * n * dm + 3 * dm * dm + q + phi
    elif kind == "train":
        # dZ from the recurrence (T - 1 products with S^T, one with B^T); dA, dV~, dQ, dK~; dK, dV
        flops += layer * T + 2 * attend + compress
        size += q + q + 2 * kv
    elif kind == "learned":
        # z B_t in every layer but the first as well, the same backwards, two products for every layer's dS_t and dB_t,
        # and the gradient of Phi
        flops += layer * (T - 1) + layer * (2 * T - 1) + 2 * attend + compress + layer * (2 * T - 1) + compress
        size += q + q + 2 * kv + 2 * T * H * d * d
        extra = 4 * (2 * T * H * d * d + T * H + phi)
    return {"bytes": size * es + extra, "flops": flops}


def tolerance(case):
    """About four times what was seen between the tensor-core and the float32 kernels on the same inputs, and between
    inputs that differ by a quarter of a bf16 step (2^-24 in float32).  In a gradient one decision taken differently in
    one of the layers moves single entries of dQ by up to their typical size."""
    train = case["pass"] in ("train", "learned")
    if case["dtype"] == "fp32":
        return {"rel": 5e-3, "max": 0.6} if train else {"rel": 5e-6, "max": 5e-5}
    return {"rel": 0.02, "max": 0.9} if train else {"rel": 0.025, "max": 0.5}


def _phi(m, n, h, dt):
    """Measurement matrix of head h for seed 0: Philox4x32-10, four Gaussians of a block by Box-Muller on 23-bit
    uniforms, divided by sqrt(m) and held in the storage type; as float64."""
    lo32 = 0xFFFFFFFF
    q = torch.arange(h * m * n // 4, ((h + 1) * m * n + 3) // 4, device="cuda")
    c = [q & lo32, q >> 32, torch.zeros_like(q), torch.zeros_like(q)]
    k = [0, 0]
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57                 # modulo 2^64
        c = [((p1 >> 32) & lo32) ^ c[1] ^ k[0], p1 & lo32, ((p0 >> 32) & lo32) ^ c[3] ^ k[1], p0 & lo32]
        k = [(k[0] + 0x9E3779B9) & lo32, (k[1] + 0xBB67AE85) & lo32]
    u = [((w >> 9).double() + 0.5) * 2.0 ** -23 for w in c]
    g = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = torch.sqrt(-2.0 * torch.log(a))
        g += [r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)]
    first = h * m * n % 4
    g = torch.stack(g, 1).flatten()[first:first + m * n] / math.sqrt(m)
    return g.to(torch.float32).to(dt).double().view(m, n)


def exact(case, seed):
    """The paper's equations in 64 bits on the same inputs: K~ = Phi K, V~ = Phi V, Z = softmax(Q K~^T / sqrt(d)) V~,
    alpha <- eta_theta(alpha S + Z B) with S = I - mu M^T M, B = mu M, M = Phi[:d, :d] Psi, 1 / mu the largest absolute
    row sum of M^T M and theta = mu lambda, out = alpha Psi^T; gradients by torch's autograd."""
    s = _inputs(case, seed)
    dt, f64 = _dtype(case), torch.float64
    B, H, n, n_q, d, m, T = (case[k] for k in ("B", "H", "n", "n_q", "d", "m", "T"))
    kind = case["pass"]
    if kind == "layer":
        QKV = (s["X"].double().view(B * n, -1) @ s["W"].double()).view(B, n, 3, H, d).permute(2, 0, 3, 1, 4)
        s["Q"], s["K"], s["V"] = QKV[0], QKV[1], QKV[2]
    eye = torch.eye(d, dtype=f64, device="cuda")
    psi = s["psi"].double() if case["psi"] else eye
    grad = kind in ("train", "learned")
    out = torch.empty(B, H, n_q, d, dtype=f64, device="cuda")
    res = {k: torch.empty(s[k].shape, dtype=f64, device="cuda") for k in "QKV"} if grad else {}
    if kind == "learned":
        res.update(S=torch.zeros(T, H, d, d, dtype=f64, device="cuda"), B=torch.zeros(T, H, d, d, dtype=f64, device="cuda"),
                   phi=torch.zeros(H, m, n, dtype=f64, device="cuda"))
    for h in range(H):
        phi = _phi(m, n, h, dt)
        M = phi[:d, :d] @ psi
        G = M.t() @ M
        mu = 1.0 / G.abs().sum(1).max()
        Ss, Bs, thetas = (eye - mu * G).expand(T, d, d), (mu * M).expand(T, d, d), (mu * case["lam"]).expand(T)
        if kind == "learned":
            Ss, Bs = ((x.float() + s[k][:, h]).to(dt).double().requires_grad_(True) for x, k in ((Ss, "dS"), (Bs, "dBm")))
            thetas = thetas * s["dtheta"][:, h].double()
            phi = s["phi"][h].double().requires_grad_(True)
        for b in range(B):
            q, k, v = (s[x][b, h].detach().double().requires_grad_(grad) for x in "QKV")
            with torch.set_grad_enabled(grad):
                z = torch.softmax(q @ (phi @ k).t() / math.sqrt(d), 1) @ (phi @ v)
                c = z @ Bs[0]
                alpha = torch.zeros_like(z)
                for t in range(T):
                    x = (z @ Bs[t] if kind == "learned" else c) + (alpha @ Ss[t] if t else 0.0)
                    alpha = x - torch.clamp(x, -thetas[t], thetas[t])
                o = alpha @ psi.t()
            out[b, h] = o.detach()
            if grad:
                of = (q, k, v) + ((Ss, Bs, phi) if kind == "learned" else ())
                gr = torch.autograd.grad(o, of, s["dOut"][b, h].double())
                for x, y in zip("QKV", gr):
                    res[x][b, h] = y
                if kind == "learned":
                    res["S"][:, h] += gr[3]
                    res["B"][:, h] += gr[4]
                    res["phi"][h] += gr[5]
    return (out,) + tuple(res.values()) if grad else out
