"""What the framework's users have it do, as measurable cases: the shearlet transform in both directions, ADMM
segmentations from one 64 x 64 image to a 2048 x 2048 RGB one, an uneven batch, a training step through the
unrolled solver, and the TV and NL-means models.  Every case runs through the public classes of
``paper_1112_1805_gb300.api`` with their default plans.

A case is a dict of plain values; its ``kind`` says which entry point it runs.  ``exact`` restates the method in
64-bit torch (Haeuser & Steidl, arXiv:1112.1805, Sec. 2-4) without the package's code.
"""

import math
import random

import numpy as np
import torch

from paper_1112_1805_gb300 import binding as B
from paper_1112_1805_gb300.api import (FilterBank, NLSegmenter, ShearletBatch, ShearletSegmenter, TVSegmenter,
                                       unrolled_segmentation)

# sides the library takes: products of powers of 2, 3 and 5
SMOOTH = sorted(n for n in {2 ** a * 3 ** b * 5 ** c for a in range(12) for b in range(8) for c in range(6)} if n <= 2048)


def listed():
    return [
        # the smallest transform: one preview-sized channel; latency and launches count
        {"name": "analyze-64", "kind": "analyze", "H": 64, "W": 64, "J": 2, "nch": 1},
        # the coefficients of four label layers of the 512 x 512 benchmark image
        {"name": "analyze-512", "kind": "analyze", "H": 512, "W": 512, "J": 4, "nch": 4},
        # synthesis of two channels at the batch's first shape (factors 3 and 5)
        {"name": "synthesize-384x640", "kind": "synthesize", "H": 384, "W": 640, "J": 4, "nch": 2},
        # synthesis of an RGB full-HD frame
        {"name": "synthesize-1080x1920", "kind": "synthesize", "H": 1080, "W": 1920, "J": 4, "nch": 3},
        # segmentation of a small image, interactive use: every launch counts
        {"name": "admm-64", "kind": "admm", "H": 64, "W": 64, "C": 1, "K": 3, "J": 2, "iters": 20},
        # the benchmark image, iterations of the main loop
        {"name": "admm-512", "kind": "admm", "H": 512, "W": 512, "C": 1, "K": 4, "J": 4, "iters": 10},
        # a VGA photograph: sides with several odd factors
        {"name": "admm-480x640", "kind": "admm", "H": 480, "W": 640, "C": 1, "K": 5, "J": 4, "iters": 5},
        # the largest image: RGB, eight colours, coefficients of 17 GB
        {"name": "admm-2048-rgb", "kind": "admm", "H": 2048, "W": 2048, "C": 3, "K": 8, "J": 5, "iters": 3},
        # images of uneven sizes and label counts solved side by side
        {"name": "batch-uneven", "kind": "batch", "n": 8, "mix": 1805, "side": 768, "iters": 5},
        # one training image: forward and backward through the unrolled solver
        {"name": "unrolled-256", "kind": "unrolled", "H": 256, "W": 256, "K": 4, "J": 3, "T": 10, "ckpt": 5},
        # the TV model on the benchmark image, the paper's 100 iterations
        {"name": "tv-512", "kind": "tv", "H": 512, "W": 512, "C": 1, "K": 4, "iters": 100, "per_label": False},
        # the NL-means model on the benchmark image: the graph of a new image and the paper's 100 iterations
        {"name": "nl-512", "kind": "nl", "H": 512, "W": 512, "C": 1, "K": 4, "iters": 100},
    ]


def scales(H, W, most=5):
    """The paper's number of scales for a size, floor(log2(min(H, W)) / 2)."""
    return max(1, min(most, int(math.floor(0.5 * math.log2(min(H, W))))))


def eta(J):
    return 2 ** (J + 2) - 3


def a_side(rng, lo, hi, step=1):
    """A legal side in [lo, hi], spread over its logarithm; step 2: twice a legal half side."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((n * step for n in SMOOTH if lo <= n * step <= hi), key=lambda n: abs(math.log(n / x)))


def draw(rng):
    kind = rng.choice(["analyze", "synthesize", "admm", "admm", "admm", "batch", "unrolled", "tv", "nl"])
    while True:
        if kind in ("analyze", "synthesize"):
            H, W = a_side(rng, 32, 2048), a_side(rng, 32, 2048, 2)
            c = {"kind": kind, "H": H, "W": W, "J": scales(H, W), "nch": rng.randint(1, 4)}
            if c["nch"] * eta(c["J"]) * H * W <= 3 * 61 * 1080 * 1920:
                return c
        elif kind == "admm":
            H, W = a_side(rng, 32, 2048), a_side(rng, 32, 2048, 2)
            c = {"kind": kind, "H": H, "W": W, "C": rng.choice([1, 1, 3]), "K": rng.randint(2, 8), "J": scales(H, W),
                 "iters": rng.randint(3, 20)}
            if c["iters"] * c["K"] * eta(c["J"]) * H * W <= 4e9:
                return c
        elif kind == "batch":
            return {"kind": kind, "n": rng.randint(3, 8), "mix": rng.randint(0, 10 ** 6),
                    "side": rng.choice([256, 512, 768]), "iters": rng.randint(3, 8)}
        elif kind == "unrolled":
            H, W = a_side(rng, 64, 512), a_side(rng, 64, 512, 2)
            c = {"kind": kind, "H": H, "W": W, "K": rng.randint(2, 5), "J": scales(H, W, 3), "T": rng.randint(4, 12),
                 "ckpt": rng.randint(2, 6)}
            if c["T"] * c["K"] * eta(c["J"]) * H * W <= 1e8:
                return c
        elif kind == "tv":
            H, W = a_side(rng, 64, 2048), a_side(rng, 64, 2048, 2)
            c = {"kind": kind, "H": H, "W": W, "C": rng.choice([1, 3]), "K": rng.randint(2, 8),
                 "iters": rng.randint(20, 100), "per_label": rng.random() < 0.25}
            if c["iters"] * c["K"] * H * W <= 4e8:
                return c
        else:
            H, W = a_side(rng, 64, 512), a_side(rng, 64, 512, 2)
            return {"kind": kind, "H": H, "W": W, "C": 1, "K": rng.randint(2, 6), "iters": rng.randint(20, 100)}


def batch_shapes(case):
    """The uneven batch's (H, W, K, J): 384 x 640 first, then sides from the framework's batch workload."""
    rng = random.Random(case["mix"])
    sides = [s for s in (128, 160, 192, 256, 320, 384, 512, 640, 768) if s <= case["side"]]
    got = [(384, 640)] if case["side"] >= 640 else []
    while len(got) < case["n"]:
        got.append((rng.choice(sides), rng.choice(sides)))
    return [(H, W, rng.randint(2, 6), scales(H, W)) for H, W in got]


def codebook(K, C):
    if C == 3:  # the colours {0.2, 0.8}^3
        return np.array([[a, b, c] for a in (0.2, 0.8) for b in (0.2, 0.8) for c in (0.2, 0.8)])[:K].astype(np.float32)
    return np.linspace(0.2, 0.8, K, dtype=np.float32)[:, None]


def weights(J):
    """0.1 (0, 0.1, 0.2, 0.4, ...), the paper's pattern of shearlet weights."""
    return np.array([0.0] + [0.01 * 2.0 ** j for j in range(J)], dtype=np.float32)


def an_image(H, W, K, C, seed):
    """Regions bounded by ellipses with their codebook value, an oriented grating per label and noise of standard
    deviation 0.05: (image [C, H, W] float32, labels [H, W])."""
    rng = np.random.RandomState(seed % (2 ** 32))
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    y = torch.arange(H, device="cuda", dtype=torch.float32)[:, None]
    x = torch.arange(W, device="cuda", dtype=torch.float32)[None, :]
    lab = torch.zeros((H, W), dtype=torch.int64, device="cuda")
    for i in range(6 + K):
        cy, cx = rng.uniform(0, H), rng.uniform(0, W)
        a, b = rng.uniform(0.1, 0.25, 2) * min(H, W)
        th, k = rng.uniform(0, math.pi), (i % K if i < K else rng.randint(0, K))
        p = (x - cx) * math.cos(th) + (y - cy) * math.sin(th)
        q = (y - cy) * math.cos(th) - (x - cx) * math.sin(th)
        lab = torch.where((p / a) ** 2 + (q / b) ** 2 <= 1.0, torch.full_like(lab, int(k)), lab)
    cb = torch.tensor(codebook(K, C), device="cuda")
    img = cb[lab].permute(2, 0, 1).contiguous()
    for k in range(K):
        th, period = k * math.pi / K, rng.uniform(8, 16)
        img = img + torch.where(lab == k, 0.15 * torch.sin((x * math.cos(th) + y * math.sin(th)) * (2 * math.pi / period)),
                                torch.zeros_like(img[0]))
    return (img + 0.05 * torch.randn((C, H, W), generator=g, device="cuda")).contiguous(), lab


def channels(case, seed):
    """`nch` image channels as a user transforms them."""
    return torch.stack([an_image(case["H"], case["W"], 4, 1, seed + 7919 * c)[0][0] for c in range(case["nch"])])


def coefficients(case, seed):
    """Coefficients as they come out of a shrinkage: mostly small, a share of them zero."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    c = torch.randn((case["nch"], eta(case["J"]), case["H"], case["W"]), generator=g, device="cuda")
    return torch.nn.functional.softshrink(c.mul_(0.05), 0.04)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("analyze", "synthesize"):
        x = channels(case, seed) if kind == "analyze" else coefficients(case, seed)
        return {"case": case, "bank": FilterBank(case["H"], case["W"], case["J"]), "x": x}
    if kind == "batch":
        shapes = batch_shapes(case)
        imgs = [an_image(H, W, K, 1, seed + 31 * i)[0] for i, (H, W, K, J) in enumerate(shapes)]
        b = ShearletBatch(imgs, [codebook(K, 1) for _, _, K, _ in shapes], [weights(J) for *_, J in shapes])
        return {"case": case, "batch": b, "host": [t.cpu().pin_memory() for t in imgs],
                "images": [b.image(i) for i in range(len(shapes))]}
    H, W, K = case["H"], case["W"], case["K"]
    f, lab = an_image(H, W, K, case.get("C", 1), seed)
    if kind == "unrolled":
        target = torch.nn.functional.one_hot(lab, K).permute(2, 0, 1).float().contiguous()
        return {"case": case, "bank": FilterBank(H, W, case["J"]), "f": f, "target": target,
                "cb": torch.tensor(codebook(K, 1), device="cuda", requires_grad=True),
                "lam": torch.tensor(weights(case["J"]), device="cuda", requires_grad=True)}
    cb = codebook(K, case["C"])
    if kind == "admm":
        bank = FilterBank(H, W, case["J"])
        return {"case": case, "f": f, "seg": ShearletSegmenter(bank, f, cb, weights(case["J"]))}
    if kind == "tv":
        return {"case": case, "f": f, "seg": TVSegmenter(f, cb, 1.0 / 12.0, 1.0, per_label=case["per_label"])}
    return {"case": case, "f": f, "seg": NLSegmenter(f, cb, 1.0 / 32.0, 0.2)}


def keeps_bv(case):
    """Whether the dual variable of the coefficients is read out as well (up to 1 GiB)."""
    return case["kind"] == "admm" and 4 * case["K"] * eta(case["J"]) * case["H"] * case["W"] <= 2 ** 30


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "analyze":
        return state["bank"].analyze(state["x"])
    if kind == "synthesize":
        return state["bank"].synthesize(state["x"])
    if kind == "batch":
        for seg, img in zip(state["images"], state["host"]):
            seg.reset(img)
        state["batch"].step(case["iters"])
        state["batch"].synchronize()
        return [seg.get(B.SEG_W) for seg in state["images"]]
    if kind == "unrolled":
        state["cb"].grad = state["lam"].grad = None
        w = unrolled_segmentation(state["f"], state["cb"], state["lam"], state["bank"], 1.0, case["T"], case["ckpt"])
        ((w - state["target"]) ** 2).mean().backward()
        return {"w": w.detach(), "codebook": state["cb"].grad, "lambda": state["lam"].grad}
    seg = state["seg"]
    seg.reset(state["f"])
    seg.step(case["iters"])
    out = {"u": seg.get(B.SEG_U), "w": seg.get(B.SEG_W), "bw": seg.get(B.SEG_BW)}
    if keeps_bv(case):
        out["bv"] = seg.get(B.SEG_BV)
    return out


def work(case):
    """Bytes that have to move and the operations of one pass.  A real 2-D transform of P values counts 2.5 P log2 P;
    the filter bank is read once a pass (once an iteration where the passes in between evict it)."""
    def transform(H, W, J, nch):
        P = H * W
        return 4.0 * P * (nch * (1 + eta(J)) + 0.5 * eta(J)), 2.5 * P * math.log2(P) * nch * (1 + eta(J)) + 2.0 * P * nch * eta(J)

    def admm(H, W, K, J, C, n):  # b_v read and written, w, b_w, s read, w, b_w, u written
        P = H * W
        by = n * (P * K * (8.0 * eta(J) + 24.0) + 2.0 * P * eta(J)) + 4.0 * P * (C + 4 * K)
        return by, n * (2 * 2.5 * P * math.log2(P) * K * (1 + eta(J)) + 12.0 * P * K * eta(J) + 20.0 * P * K)

    kind = case["kind"]
    if kind in ("analyze", "synthesize"):
        by, fl = transform(case["H"], case["W"], case["J"], case["nch"])
    elif kind == "admm":
        by, fl = admm(case["H"], case["W"], case["K"], case["J"], case["C"], case["iters"])
        by += 8.0 * case["K"] * case["H"] * case["W"] * (3 + (eta(case["J"]) if keeps_bv(case) else 0))
    elif kind == "batch":
        got = [admm(H, W, K, J, 1, case["iters"]) for H, W, K, J in batch_shapes(case)]
        by, fl = sum(g[0] for g in got), sum(g[1] for g in got)
    elif kind == "unrolled":  # the forward and the adjoint sweep
        by, fl = admm(case["H"], case["W"], case["K"], case["J"], 1, 2 * case["T"])
    else:
        P, K, n = case["H"] * case["W"], case["K"], case["iters"]
        if kind == "tv":  # b_v (2), w, b_w, s read; b_v, w, b_w, u written
            by, fl = n * P * K * 4.0 * 9 + 4.0 * P * (case["C"] + 7 * K), n * P * K * (5.0 * math.log2(P) + 40.0)
        else:  # 10 neighbours: b_v read and written, 54 steps of the solve on vectors that stay on the chip
            by = n * (P * K * 4.0 * (2 * 10 + 6) + P * 2.0 * 10) + 4.0 * P * (case["C"] + 7 * K)
            fl = n * P * K * (54 * 28.0 + 120.0) + P * 224 * 25 * 4.0 * case["C"]
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------------------------------------------
# The same in 64 bits.
# ---------------------------------------------------------------------------------------------------------------


def _v(x):
    x = x.clamp(0.0, 1.0)
    return x ** 4 * (35.0 + x * (-84.0 + x * (70.0 - 20.0 * x)))


def _b(x):
    a = x.abs()
    up, down = torch.sin(0.5 * math.pi * _v(a - 1.0)), torch.cos(0.5 * math.pi * _v(0.5 * a - 1.0))
    return torch.where((a < 1.0) | (a > 4.0), torch.zeros_like(a), torch.where(a <= 2.0, up, down))


def _psi1(w):
    return torch.sqrt(_b(2.0 * w) ** 2 + _b(w) ** 2)


def _psi2(w):
    return torch.sqrt(_v(torch.where(w <= 0.0, 1.0 + w, 1.0 - w)))


def bank64(H, W, J):
    """The filters' half spectra, one at a time: low-pass; per scale the horizontal shears, the vertical ones and the
    two glued ones; on Nyquist lines the root mean square of a filter and its mirror image."""
    def freq(N):
        n = torch.arange(N, device="cuda", dtype=torch.float64)
        return torch.where(n < (N + 1) // 2, n, n - N)

    w1, w2 = freq(H)[:, None].expand(H, W), freq(W)[None, :].expand(H, W)
    a1, a2 = w1.abs() * W, w2.abs() * H
    ch, cv, seam = a2 < a1, a1 < a2, (a1 == a2) & (a1 > 0)
    zero = torch.zeros((H, W), dtype=torch.float64, device="cuda")

    def part(j, k, horizontal):
        s = 4.0 ** (J - j)
        num, den = (w2 * H, w1 * W) if horizontal else (w1 * W, w2 * H)
        r = num / torch.where(den == 0, torch.ones_like(den), den)
        return _psi1(w1 * s / H if horizontal else w2 * s / W) * _psi2(r * 2.0 ** j + k)

    def half(a):
        m = torch.roll(a.flip(0, 1), (1, 1), (0, 1))
        nyq = torch.zeros((H, W), dtype=torch.bool, device="cuda")
        if H % 2 == 0:
            nyq[H // 2] = True
        nyq[:, W // 2] = True
        return torch.where(nyq, torch.sqrt(0.5 * (a * a + m * m)), a)[:, : W // 2 + 1].contiguous()

    low = torch.maximum((w1 * 4.0 ** J / H).abs(), (w2 * 4.0 ** J / W).abs())
    yield half(torch.where(low <= 0.5, torch.ones_like(low),
                           torch.where(low < 1.0, torch.cos(0.5 * math.pi * _v(2.0 * low - 1.0)), zero)))
    for j in range(J):
        n = 2 ** j
        for k in range(-n + 1, n):
            yield half(torch.where(ch, part(j, k, True), zero))
        for k in range(-n + 1, n):
            yield half(torch.where(cv, part(j, k, False), zero))
        for k in (-n, n):
            yield half(torch.where(ch | seam, part(j, k, True), torch.where(cv, part(j, k, False), zero)))


def simplex(g):
    """Projection of the values along axis 0 onto the unit simplex."""
    K = g.shape[0]
    c = (torch.cumsum(torch.sort(g, dim=0, descending=True)[0], 0) - 1.0)
    n = torch.arange(1, K + 1, device=g.device, dtype=g.dtype).reshape((K,) + (1,) * (g.dim() - 1))
    return (g - (c / n).max(0, keepdim=True)[0]).clamp_min(0.0)


def data_term(f, cb):
    return ((f.double()[None] - cb[:, :, None, None]) ** 2).sum(1)


def admm64(f, cb, lam, gamma, J, n, grad=False):
    """n iterations from zero: (u, w, b_w, b_v or None); with `grad` on out-of-place operations only."""
    H, W = f.shape[-2:]
    K, P = cb.shape[0], H * W
    s = data_term(f, cb)
    bank = torch.stack(list(bank64(H, W, J)))
    t = torch.stack([gamma * lam[j] for j in [0] + [j + 1 for j in range(J) for _ in range(4 * 2 ** j)]])
    w, bw, stv = torch.zeros_like(s), torch.zeros_like(s), torch.zeros_like(s)
    bv = [None] * K
    step = max(1, int(2 ** 28 // P))  # filters at a time
    for _ in range(n):
        u = 0.5 * (stv + (w - bw) - gamma * s)
        new = []
        for k in range(K):
            uh = torch.fft.rfft2(u[k])
            acc, parts = None, []
            for a in range(0, bank.shape[0], step):
                wf, th = bank[a:a + step], t[a:a + step, None, None]
                g = torch.fft.irfft2(wf * uh, s=(H, W))
                if bv[k] is not None:
                    g = g + bv[k][a // step]
                b = torch.where(g.abs() < th, g, torch.sign(g) * th)
                parts.append(b)
                z = (wf * torch.fft.rfft2(g - 2.0 * b)).sum(0)
                acc = z if acc is None else acc + z
            if not grad:
                bv[k] = None
            bv[k] = parts
            new.append(torch.fft.irfft2(acc, s=(H, W)))
        stv = torch.stack(new)
        g = bw + u
        w = simplex(g)
        bw = g - w
    return u, w, bw, bv


def tv64(f, cb, lam, gamma, n, per_label):
    H, W = f.shape[-2:]
    s = data_term(f, cb)
    y = torch.arange(H, device="cuda", dtype=torch.float64)[:, None]
    x = torch.arange(W // 2 + 1, device="cuda", dtype=torch.float64)[None, :]
    sym = 1.0 / (1.0 + 4.0 * torch.sin(math.pi * y / H) ** 2 + 4.0 * torch.sin(math.pi * x / W) ** 2)
    w, bw = torch.zeros_like(s), torch.zeros_like(s)
    b0, b1, d0, d1 = (torch.zeros_like(s) for _ in range(4))
    t = gamma * lam
    for _ in range(n):
        rhs = (w - bw) - gamma * s + (d0.roll(1, 1) - d0) + (d1.roll(1, 2) - d1)
        u = torch.fft.irfft2(sym * torch.fft.rfft2(rhs), s=(H, W))
        g0, g1 = b0 + u.roll(-1, 1) - u, b1 + u.roll(-1, 2) - u
        n2 = g0 * g0 + g1 * g1
        m = torch.sqrt(n2 if per_label else n2.sum(0, keepdim=True))
        fac = torch.where(m > t, t / m.clamp_min(1e-300), torch.ones_like(m))
        b0, b1 = fac * g0, fac * g1
        d0, d1 = g0 - 2.0 * b0, g1 - 2.0 * b1
        g = bw + u
        w = simplex(g)
        bw = g - w
    return u, w, bw


def graph64(f, p=5, window=15, a=2.0, mt=5):
    """The symmetric neighbour lists of Sec. 4, [P][2 mt] in increasing order padded with -1."""
    C, H, W = f.shape
    h, r, m = p // 2, window // 2, 2 * mt
    P = H * W
    G = np.array([[math.exp(-(i * i + j * j) / (2.0 * a * a)) for j in range(-h, h + 1)] for i in range(-h, h + 1)])
    G = G / sum(G.reshape(-1).tolist())
    fp = torch.nn.functional.pad(f.double()[None], (h, h, h, h), mode="reflect")[0]
    big = torch.full((C, H + 2 * (h + r), W + 2 * (h + r)), math.inf, dtype=torch.float64, device="cuda")
    big[:, r:r + H + 2 * h, r:r + W + 2 * h] = fp
    dist = torch.full((window * window, H, W), math.inf, dtype=torch.float64, device="cuda")
    yy, xx = torch.arange(H, device="cuda")[:, None], torch.arange(W, device="cuda")[None, :]
    for c in range(window * window):
        dy, dx = c // window - r, c % window - r
        if dy == 0 and dx == 0:
            continue
        acc = torch.zeros((H, W), dtype=torch.float64, device="cuda")
        for i in range(p):
            for j in range(p):
                d = fp[:, i:i + H, j:j + W] - big[:, i + r + dy:i + r + dy + H, j + r + dx:j + r + dx + W]
                acc = acc + float(G[i, j]) * (d * d).sum(0)
        inside = (yy + dy >= 0) & (yy + dy < H) & (xx + dx >= 0) & (xx + dx < W)
        dist[c] = torch.where(inside, acc, dist[c])
    keep = 100
    val, order = torch.sort(dist.reshape(window * window, P).t().contiguous(), dim=1, stable=True)
    order = torch.where(torch.isinf(val), torch.full_like(order, -1), order)[:, :keep].cpu().tolist()
    nb, deg = [[] for _ in range(P)], [0] * P
    step = [(c // window - r) * W + (c % window - r) for c in range(window * window)]
    for i in range(P):
        left, mine = min(mt, m - deg[i]), nb[i]
        for c in order[i] if left > 0 else ():
            if c < 0:
                break
            j = i + step[c]
            if deg[j] >= m or j in mine:
                continue
            mine.append(j)
            nb[j].append(i)
            deg[i] += 1
            deg[j] += 1
            left -= 1
            if left == 0:
                break
    out = np.full((P, m), -1, dtype=np.int64)
    for i in range(P):
        out[i, : deg[i]] = sorted(nb[i])
    return torch.from_numpy(out).cuda()


def nl64(f, cb, lam, gamma, n):
    H, W = f.shape[-2:]
    K, P = cb.shape[0], H * W
    nb = graph64(f)
    m = nb.shape[1]
    has = (nb >= 0)
    to = nb.clamp_min(0)
    deg = has.sum(1).double()
    # the position of i in the list of its b-th neighbour
    rev = (nb[to] == torch.arange(P, device="cuda")[:, None, None]).double().argmax(2)
    hd = has.double()
    s = data_term(f, cb).reshape(K, P).t().contiguous()  # pixel-major [P][K]

    def gathered(x):
        return (x[to] * hd[:, :, None]).sum(1)

    def apply(x):
        return x + 2.0 * (deg[:, None] * x - gathered(x))

    u, w, bw = torch.zeros_like(s), torch.zeros_like(s), torch.zeros_like(s)
    bv = torch.zeros((P, m, K), dtype=torch.float64, device="cuda")
    d = torch.zeros_like(bv)
    flat = to * m + rev
    t = gamma * lam
    for _ in range(n):
        back = d.reshape(P * m, K)[flat] - d
        rhs = (w - bw) - gamma * s + (back * hd[:, :, None]).sum(1)
        res = rhs - apply(u)  # conjugate gradients, every label at once
        q = res.clone()
        rr = (res * res).sum(0)
        for _ in range(70):
            aq = apply(q)
            al = rr / (q * aq).sum(0).clamp_min(1e-300)
            u = u + al * q
            res = res - al * aq
            new = (res * res).sum(0)
            q = res + (new / rr.clamp_min(1e-300)) * q
            rr = new
        g = bv + (u[to] - u[:, None, :]) * hd[:, :, None]
        nrm = torch.sqrt((g * g).sum((1, 2)))
        fac = torch.where(nrm > t, t / nrm.clamp_min(1e-300), torch.ones_like(nrm))
        bv = fac[:, None, None] * g
        d = g - 2.0 * bv
        gw = bw + u
        w = simplex(gw.t()).t()
        bw = gw - w
    return tuple(v.t().reshape(K, H, W).contiguous() for v in (u, w, bw))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("analyze", "synthesize"):
        H, W, nch = case["H"], case["W"], case["nch"]
        if kind == "analyze":
            uh = torch.fft.rfft2(channels(case, seed).double())
            out = torch.empty((nch, eta(case["J"]), H, W), dtype=torch.float64, device="cuda")
            for i, wf in enumerate(bank64(H, W, case["J"])):
                out[:, i] = torch.fft.irfft2(wf * uh, s=(H, W))
            return out
        x, acc = coefficients(case, seed), 0.0
        for i, wf in enumerate(bank64(H, W, case["J"])):
            acc = acc + wf * torch.fft.rfft2(x[:, i].double())
        return torch.fft.irfft2(acc, s=(H, W))
    if kind == "batch":
        out = []
        for i, (H, W, K, J) in enumerate(batch_shapes(case)):
            f = an_image(H, W, K, 1, seed + 31 * i)[0]
            out.append(admm64(f, torch.tensor(codebook(K, 1), device="cuda").double(),
                              torch.tensor(weights(J), device="cuda").double(), 1.0, J, case["iters"])[1])
        return out
    H, W, K = case["H"], case["W"], case["K"]
    f, lab = an_image(H, W, K, case.get("C", 1), seed)
    cb = torch.tensor(codebook(K, case.get("C", 1)), device="cuda").double()
    if kind == "unrolled":
        cb.requires_grad_(True)
        lam = torch.tensor(weights(case["J"]), device="cuda").double().requires_grad_(True)
        w = admm64(f, cb, lam, 1.0, case["J"], case["T"], grad=True)[1]
        target = torch.nn.functional.one_hot(lab, K).permute(2, 0, 1).double()
        ((w - target) ** 2).mean().backward()
        return {"w": w.detach(), "codebook": cb.grad, "lambda": lam.grad}
    if kind == "admm":
        lam = torch.tensor(weights(case["J"]), device="cuda").double()
        u, w, bw, bv = admm64(f, cb, lam, 1.0, case["J"], case["iters"])
        out = {"u": u, "w": w, "bw": bw}
        if keeps_bv(case):
            out["bv"] = torch.stack([torch.cat(p) for p in bv])
        return out
    if kind == "tv":
        u, w, bw = tv64(f, cb, 1.0 / 12.0, 1.0, case["iters"], case["per_label"])
    else:
        u, w, bw = nl64(f, cb, 1.0 / 32.0, 0.2, case["iters"])
    return {"u": u, "w": w, "bw": bw}
