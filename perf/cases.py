"""The work this library is measured on: one SSBA layer of a DiT as a program calls it, from the
smallest image to 4K, forward and backward, with its upstream projection and the VAE's wavelets.

Every case goes through ``paper_2605_15684_gb300.api`` with the arguments a program passes: it
holds a descriptor, its inputs and (for the projection) its weights, lets the calls allocate
their outputs, and uses the default workspace. Image sizes follow the model's geometry (8x VAE,
2x2 patchify: a P pixel side is P / 16 tokens, blocks are 8x8 tokens).
"""
import math

import torch
import torch.nn.functional as F

from paper_2605_15684_gb300 import api

BF16, FP32 = "bf16", "fp32"
_DT = {BF16: torch.bfloat16, FP32: torch.float32}


def _layer(kind, B, heads, H, W, shift, rho, dtype=BF16, **more):
    return dict(kind=kind, B=B, heads=heads, H=H, W=W, shift=shift, rho=rho, dtype=dtype, **more)


def listed():
    return [
        # A 256 px preview of one layer: the smallest call, where launches and the host count.
        dict(_layer("fused", 1, 24, 16, 16, 4, 0.75), name="layer_256px"),
        # 512 px generation, the mask and the attention as two calls (a program that keeps the lists).
        dict(_layer("two_calls", 1, 24, 32, 32, 0, 0.8416), name="layer_512px"),
        # 1024 px generation, a shifted layer in one call: the benchmark's layer.
        dict(_layer("fused", 1, 24, 64, 64, 4, 0.8416), name="layer_1024px"),
        # A batch of four 1024 px images at the uniform 75 % ratio.
        dict(_layer("fused", 4, 24, 64, 64, 0, 0.75), name="layer_1024px_b4"),
        # A wide image with a text prompt (333 tokens) attended by every query block.
        dict(_layer("text", 1, 24, 48, 88, 4, 0.8416, T_txt=333), name="layer_wide_text"),
        # 2048 px, the largest square image of the model.
        dict(_layer("fused", 1, 24, 128, 128, 4, 0.84), name="layer_2048px"),
        # A 4K frame (240 x 136 tokens, 510 blocks a head): the longest rows, two calls.
        dict(_layer("two_calls", 1, 24, 136, 240, 4, 0.75), name="layer_4k"),
        # Dense attention of a 1024 px layer (0 % sparsity, the layers a schedule leaves dense).
        dict(_layer("dense", 1, 24, 64, 64, 0, 0.0), name="dense_1024px"),
        # A training step of one layer: forward with its lists, then every gradient.
        dict(_layer("train", 1, 24, 64, 64, 4, 0.8416), name="train_1024px"),
        # The same in fp32 with a shift that is no multiple of 4 (validation of a model's gradients).
        dict(_layer("train", 1, 24, 32, 32, 3, 0.8416, FP32), name="train_fp32_512px"),
        # The layer's QKV projection with RoPE and block means, and the lists from those means.
        dict(_layer("project", 1, 24, 64, 64, 4, 0.8416, bias=True), name="project_1024px"),
        # Encoder and decoder wavelet pyramids of the f8 VAE over a 1024 px feature map.
        dict(kind="haar", N=1, C=128, H=1024, W=1024, levels=3, nb=4, dtype=BF16, name="haar_1024px"),
    ]


# ----------------------------------------------------------------------------- more of the same
_MOST_FLOPS = 1.6e12  # of the largest listed case


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, lo, hi):
    """Blocks (rows, columns) with lo..hi blocks in all and sides at most 1 : 2.5."""
    while True:
        area, aspect = _log(rng, lo, hi), _log(rng, 0.4, 2.5)
        r, c = round(math.sqrt(area * aspect)), round(math.sqrt(area / aspect))
        if r >= 2 and c >= 2 and lo <= r * c <= hi:
            return r, c


def draw(rng):
    kind = rng.choice(["fused", "fused", "two_calls", "two_calls", "text", "dense", "train", "train", "train32",
                       "project", "haar"])
    if kind == "haar":
        L = rng.choice([1, 2, 3])
        m = 1 << L
        return dict(kind="haar", N=rng.choice([1, 2]), C=int(_log(rng, 8, 128)), H=m * int(_log(rng, 64, 1024) / m),
                    W=m * int(_log(rng, 64, 1024) / m), levels=L, nb=rng.choice([3, 4]), dtype=rng.choice([BF16, FP32]))
    while True:
        lo, hi = {"train32": (4, 36), "two_calls": (4, 510)}.get(kind, (4, 256))
        r, c = _grid(rng, lo, hi)
        heads = rng.choice([12, 16, 24])
        B = rng.choice([1, 1, 2, 4]) if kind != "train32" else 1
        rho = 0.0 if kind == "dense" else rng.choice([0.5, 0.75, 0.8416, 0.9])
        shift = rng.choice([0, 4])
        if kind == "train32":
            case = _layer("train", B, heads, 8 * r, 8 * c, rng.choice([0, 3, 4]), rho, FP32)
        elif kind == "text":
            case = _layer(kind, B, heads, 8 * r, 8 * c, shift, rho, T_txt=int(_log(rng, 8, 1024)))
        elif kind == "project":
            case = _layer(kind, B, heads, 8 * r, 8 * c, shift, rho, bias=rng.random() < 0.5)
        else:
            case = _layer(kind, B, heads, 8 * r, 8 * c, shift, rho)
        if work(case)["flops"] * (1.4 if kind == "train" else 1.0) <= _MOST_FLOPS:
            return case


# ----------------------------------------------------------------------------- a program's inputs
def _desc(c):
    return api.SsbaDesc(c["B"], c["heads"], c["H"], c["W"], shift_r=c["shift"], shift_c=c["shift"], rho=c["rho"],
                        dtype=_DT[c["dtype"]])


def _keep(c):
    Tb = c["H"] * c["W"] // 64
    return Tb - int(math.floor(Tb * c["rho"]))


def _tokens(g, field, c):
    """Image tokens [B, heads, N, 64]: a part that varies slowly over the grid, so that near
    blocks resemble each other as they do in an image, and detail of its own per token."""
    n = torch.randn(c["B"], c["heads"], c["H"] * c["W"], 64, generator=g, device="cuda")
    return n.mul_(0.87).add_(field, alpha=0.6).to(_DT[c["dtype"]])


def _inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    coarse = torch.randn(c["B"] * c["heads"], 64, max(2, c["H"] // 16), max(2, c["W"] // 16), generator=g, device="cuda")
    f = F.interpolate(coarse, size=(c["H"], c["W"]), mode="bilinear", align_corners=True)
    f = f.reshape(c["B"], c["heads"], 64, -1).transpose(2, 3).contiguous()
    return g, f


def prepare(case, seed):
    c = case
    if c["kind"] == "haar":
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        x = torch.randn(c["N"], c["C"], c["H"], c["W"], generator=g, device="cuda").to(_DT[c["dtype"]])
        return dict(c=c, x=x)
    if c["kind"] == "project":
        g = torch.Generator(device="cuda").manual_seed(int(seed))
        Dm = c["heads"] * 64
        X = torch.randn(c["B"], c["H"] * c["W"], Dm, generator=g, device="cuda").bfloat16()
        Wqkv = (torch.randn(3 * Dm, Dm, generator=g, device="cuda") / math.sqrt(Dm)).bfloat16()
        bias = torch.randn(3 * Dm, generator=g, device="cuda") * 0.1 if c["bias"] else None
        return dict(c=c, desc=_desc(c), X=X, W=Wqkv, bias=bias)
    g, field = _inputs(c, seed)
    s = dict(c=c, desc=_desc(c), Q=_tokens(g, field, c), K=_tokens(g, field, c), V=_tokens(g, field, c))
    del field
    if c["kind"] == "train":
        s["dO"] = torch.randn(s["Q"].shape, generator=g, device="cuda").to(_DT[c["dtype"]])
    if c["kind"] == "text":
        shp = (c["B"], c["heads"], c["T_txt"], 64)
        s["Kt"], s["Vt"] = (torch.randn(shp, generator=g, device="cuda").bfloat16() for _ in range(2))
    return s


# ----------------------------------------------------------------------------- one pass
def run(s):
    c = s["c"]
    kind = c["kind"]
    if kind == "haar":
        ys = api.haar_dwt_pyramid(s["x"], c["levels"], nb=c["nb"])
        return ys, api.haar_iwt_pyramid(ys, c["C"], nb=c["nb"])
    d = s["desc"]
    if kind == "project":
        Q, K, V, qb, kb = api.qkv_rope_pool(d, s["X"], s["W"], s["bias"])
        idx, cnt = api.select_mask(d, qb, kb)
        return Q, K, V, qb, kb, idx, cnt
    Q, K, V = s["Q"], s["K"], s["V"]
    if kind == "fused":
        O, lse, idx, cnt, qb, kb = api.forward_fused(d, Q, K, V)
        return O, lse, idx, cnt, qb, kb
    if kind == "dense":
        return api.forward_dense(d, Q, K, V)
    idx, cnt = api.build_mask(d, Q, K)
    if kind == "text":
        O, lse = api.forward_joint(d, Q, K, V, s["Kt"], s["Vt"], idx, cnt)
        return O, lse, idx, cnt
    O, lse = api.forward(d, Q, K, V, idx, cnt)
    if kind == "two_calls":
        return O, lse, idx, cnt
    dQ, dK, dV = api.backward(d, Q, K, V, O, lse, s["dO"], idx, cnt)
    return O, lse, dQ, dK, dV, idx, cnt


def work(case):
    c = case
    es = 2 if c["dtype"] == BF16 else 4
    if c["kind"] == "haar":
        n = c["N"] * c["C"] * c["H"] * c["W"]
        bands = [n // 4 ** l * c["nb"] for l in range(1, c["levels"] + 1)]  # of each level
        details = [n // 4 ** l * (c["nb"] - 1) for l in range(1, c["levels"])] + [bands[-1]]  # read by the inverse
        return {"bytes": es * (n + sum(bands) + sum(details) + n), "flops": 8 * n}
    BH, N, d = c["B"] * c["heads"], c["H"] * c["W"], 64
    Tb = N // 64
    keep = Tb if c["kind"] == "dense" else _keep(c)
    tok = BH * N * d * es  # one of Q, K, V, O
    lists = 4 * BH * Tb * (keep + 1)
    means = 2 * 4 * BH * Tb * d
    if c["kind"] == "project":
        Dm = c["heads"] * 64
        return {"bytes": es * (c["B"] * N * Dm + 3 * Dm * Dm) + 3 * tok + means + lists,
                "flops": 2 * c["B"] * N * Dm * 3 * Dm + 2 * BH * Tb * Tb * d}
    attend = 4 * BH * N * d * 64 * keep + 4 * BH * N * d * c.get("T_txt", 0)
    select = 0 if c["kind"] == "dense" else 2 * BH * Tb * Tb * d
    if c["kind"] == "train":  # the gradients: five products where the forward has two
        return {"bytes": 5 * tok + 4 * BH * N + lists + 3 * 4 * BH * N * d, "flops": int(3.5 * attend) + select}
    b = 4 * tok + 4 * BH * N + (lists if select else 0) + (means if c["kind"] == "fused" else 0)
    return {"bytes": b + 2 * BH * c.get("T_txt", 0) * d * es, "flops": attend + select}


def tolerance(case):
    """About four times the distance from exact() that one pass shows: 1.7e-3 for bf16 results
    (3.3e-3 for dQ, which also takes O as it was rounded), 5e-7 to 1.1e-6 for fp32 ones. Lists
    are whole numbers that only a tie within the rounding of a score can change."""
    if case["dtype"] == FP32:
        return {"rel": 1e-6 if case["kind"] == "haar" else 5e-6, "differ": 1e-3}
    return {"rel": 1.3e-2 if case["kind"] == "train" else 7e-3, "differ": 1e-3}


# ----------------------------------------------------------------------------- the same in 64 bits
def _to_blocks(x, c):
    """[..., N, d] -> [..., Tb, 64, d]: the 8x8 blocks of the rolled grid."""
    H, W, s = c["H"], c["W"], c["shift"]
    y = torch.roll(x.reshape(*x.shape[:-2], H, W, x.shape[-1]), (s, s), (-3, -2))
    y = y.reshape(*x.shape[:-2], H // 8, 8, W // 8, 8, x.shape[-1]).transpose(-4, -3)
    return y.reshape(*x.shape[:-2], H * W // 64, 64, x.shape[-1])


def _from_blocks(y, c):
    H, W, s = c["H"], c["W"], c["shift"]
    x = y.reshape(*y.shape[:-3], H // 8, W // 8, 8, 8, y.shape[-1]).transpose(-4, -3)
    x = torch.roll(x.reshape(*y.shape[:-3], H, W, y.shape[-1]), (-s, -s), (-3, -2))
    return x.reshape(*y.shape[:-3], H * W, y.shape[-1])


def _gate(qb, kb, keep):
    S = qb @ kb.transpose(-1, -2)
    return torch.sort(torch.topk(S, keep, dim=-1).indices, dim=-1).values


def _exact_head(c, q, k, v, kt, vt, dO, idx):
    """One (batch, head) in blocks, float64: O, lse, and the gradients for dO."""
    Tb, keep = idx.shape
    scale = 1.0 / 8.0
    O, lse = torch.empty_like(q), q.new_empty(Tb, 64, 1)
    grads = [torch.zeros_like(q) for _ in range(3)] if dO is not None else None
    step = max(1, 2 ** 24 // (keep * 64 * 64))
    for a in range(0, Tb, step):
        rows = idx[a:a + step]
        kk, vv = (t[rows].flatten(1, 2) for t in (k, v))  # [n, keep * 64, d]
        if kt is not None:
            kk, vv = (torch.cat([t.expand(len(rows), -1, -1), u], 1) for t, u in ((kt, kk), (vt, vv)))
        s = (q[a:a + step] @ kk.transpose(1, 2)).mul_(scale)
        z = torch.logsumexp(s, -1, keepdim=True)
        p = (s - z).exp_()
        o = p @ vv
        O[a:a + step], lse[a:a + step] = o, z
        if dO is not None:
            g = dO[a:a + step]
            ds = (g @ vv.transpose(1, 2)).sub_((g * o).sum(-1, keepdim=True)).mul_(p).mul_(scale)
            grads[0][a:a + step] = ds @ kk
            for n, m, r in ((1, ds, q[a:a + step]), (2, p, g)):
                grads[n].index_add_(0, rows.flatten(), (m.transpose(1, 2) @ r).reshape(-1, 64, 64))
    return O, lse, grads


def _exact_attention(c, s):
    kind, B, h, N = c["kind"], c["B"], c["heads"], c["H"] * c["W"]
    if kind == "dense":
        c = dict(c, shift=0)
    keep = N // 64 if kind == "dense" else _keep(c)
    shape = (B, h, N, 64)
    O, lse = torch.empty(shape, dtype=torch.float64, device="cuda"), torch.empty(shape[:3], dtype=torch.float64, device="cuda")
    G = [torch.empty_like(O) for _ in range(3)] if kind == "train" else None
    idx = torch.empty(B, h, N // 64, keep, dtype=torch.int32, device="cuda")
    means = [torch.empty(B, h, N // 64, 64, dtype=torch.float64, device="cuda") for _ in range(2)]
    for b in range(B):
        for i in range(h):
            q, k, v = (_to_blocks(s[n][b, i].double(), c) for n in "QKV")
            kt, vt = (s[n][b, i].double() for n in ("Kt", "Vt")) if kind == "text" else (None, None)
            dO = _to_blocks(s["dO"][b, i].double(), c) if kind == "train" else None
            means[0][b, i], means[1][b, i] = q.mean(1), k.mean(1)
            rows = _gate(q.mean(1), k.mean(1), keep)
            idx[b, i] = rows
            o, z, g = _exact_head(c, q, k, v, kt, vt, dO, rows)
            O[b, i], lse[b, i] = _from_blocks(o, c), _from_blocks(z, c)[..., 0]
            for t, u in zip(G or (), g or ()):
                t[b, i] = _from_blocks(u, c)
    cnt = torch.full((B, h, N // 64), keep, dtype=torch.int32, device="cuda")
    if kind == "dense":
        return O, lse
    if kind == "fused":
        return O, lse, idx, cnt, means[0], means[1]
    return (O, lse, *G, idx, cnt) if kind == "train" else (O, lse, idx, cnt)


def _rope(x, c):
    """[B, heads, N, 64] float64: dimensions [0, 32) turn with the token's row, [32, 64) with its column."""
    n = torch.arange(c["H"] * c["W"], device="cuda")
    theta = 10000.0 ** (-torch.arange(16, dtype=torch.float64, device="cuda") / 16)
    a = torch.cat([(n // c["W"])[:, None] * theta, (n % c["W"])[:, None] * theta], 1)  # [N, 32] pairs
    e, o = x[..., 0::2], x[..., 1::2]
    return torch.stack([e * a.cos() - o * a.sin(), e * a.sin() + o * a.cos()], -1).flatten(-2)


def _exact_project(c, s):
    B, h, N = c["B"], c["heads"], c["H"] * c["W"]
    y = s["X"].double() @ s["W"].double().T
    if s["bias"] is not None:
        y = y + s["bias"].double()
    Q, K, V = (t.reshape(B, N, h, 64).transpose(1, 2) for t in y.split(h * 64, -1))
    Q, K, V = _rope(Q, c), _rope(K, c), V.contiguous()
    qb, kb = (_to_blocks(t, c).mean(-2) for t in (Q, K))
    return Q, K, V, qb, kb, None, None  # the lists follow from means of rounded values


def _exact_haar(c, x):
    n, ys, ll = c["nb"], [], x.double()
    for _ in range(c["levels"]):
        p, q, r, t = ll[..., 0::2, 0::2], ll[..., 0::2, 1::2], ll[..., 1::2, 0::2], ll[..., 1::2, 1::2]
        bands = [(p + q + r + t) / 2, (p - q + r - t) / 2, (p + q - r - t) / 2, (p - q - r + t) / 2][:n]
        ys.append(torch.cat(bands, 1))
        ll = bands[0]
    rec = ys[-1][:, :c["C"]]
    for y in reversed(ys):
        b = [rec] + list(y.split(c["C"], 1))[1:]
        hh = b[3] if n == 4 else torch.zeros_like(rec)
        ll, hl, lh = b[:3]
        rec = torch.stack([torch.stack([ll + hl + lh + hh, ll - hl + lh - hh], -1),
                           torch.stack([ll + hl - lh - hh, ll - hl - lh + hh], -1)], -3) / 2
        rec = rec.flatten(-2).flatten(-3, -2)
    return ys, rec


def exact(case, seed):
    s = prepare(case, seed)
    if case["kind"] == "haar":
        return _exact_haar(case, s["x"])
    if case["kind"] == "project":
        return _exact_project(case, s)
    return _exact_attention(case, s)
