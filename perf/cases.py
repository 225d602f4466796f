"""Performance cases: the calls that a user of the library makes, each through
``paper_1312_4746_gb300.Context``, over the sizes of the repository's own
workloads (96 x 64 with 300 samples per label up to 1024 x 1024 with 20000).

Inputs follow ``synth``'s recipe (Voronoi cells of gratings and checkerboards
times a tint plus noise; random-walk brush strokes inside each cell; Gaussian
operator rows of unit length; a Gaussian mask), drawn on the GPU from the seed
so that they are quick to make. ``exact`` restates every call in float64 torch.
"""
import math
import random

import numpy as np
import torch

import paper_1312_4746_gb300 as cs

DEV = "cuda:0"
PRECISION = {"fp32": cs.FP32, "bf16": cs.BF16, "fp8": cs.FP8}
MODE = {"persample": cs.MODE_PERSAMPLE, "factorised": cs.MODE_FACTORISED, "smooth": cs.MODE_SMOOTH}
TAU, SIGMA_C2, ALPHA, D_MIN, KAPPA, IOTA_SIGMA = 0.1, 1.3, 1.3, 1.0, 1.0, 0.01
UNSUP_SIGMA_C2, UNSUP_BETA = 0.02, 0.5  # the unsupervised mode's settings in the benchmark

_context = None


def context():
    """One context per process, as a program keeps it."""
    global _context
    if _context is None:
        _context = cs.Context(0)
    return _context


# ------------------------------------------------------------------ the cases


def listed():
    return [
        # smallest call: the 96 x 64 workload in the default (plain FP32) form,
        # an interactive scribble update where launches count; all outputs
        {"name": "data_term_fp32_96x64", "kind": "data_term", "W": 96, "H": 64, "n_labels": 3,
         "m": 300, "p": 5, "k": 50, "precision": "fp32", "mode": "persample", "all_outputs": True},
        # the default form on an ordinary (benchmark-size) image
        {"name": "data_term_fp32_481x321", "kind": "data_term", "W": 481, "H": 321, "n_labels": 5,
         "m": 2000, "p": 7, "k": 98, "precision": "fp32", "mode": "persample",
         "all_outputs": False},
        # the benchmark's headline: one image in the FP8 tensor-core form
        {"name": "data_term_fp8_481x321", "kind": "data_term", "W": 481, "H": 321, "n_labels": 5,
         "m": 2000, "p": 7, "k": 98, "precision": "fp8", "mode": "persample",
         "all_outputs": False},
        # BF16 tensor cores, the factorised likelihood, odd sizes and uneven
        # scribbles (m is the largest label's count), all outputs
        {"name": "data_term_bf16_factorised_333x247", "kind": "data_term", "W": 333, "H": 247,
         "n_labels": 4, "m": 3100, "p": 7, "k": 98, "precision": "bf16", "mode": "factorised",
         "all_outputs": True, "uneven": True},
        # the smooth co-sparse texture on the benchmark image
        {"name": "data_term_smooth_481x321", "kind": "data_term", "W": 481, "H": 321,
         "n_labels": 5, "m": 2000, "p": 7, "k": 98, "precision": "fp8", "mode": "smooth",
         "all_outputs": False},
        # the largest single image that runs in a few tens of milliseconds
        {"name": "data_term_fp8_1024x1024", "kind": "data_term", "W": 1024, "H": 1024,
         "n_labels": 10, "m": 20000, "p": 7, "k": 98, "precision": "fp8", "mode": "persample",
         "all_outputs": False},
        # codes and co-supports alone (9 x 9 patches, 162 operator rows): the
        # inputs of cs_likelihood and of the surrogate
        {"name": "codes_p9_1023x769", "kind": "codes", "W": 1023, "H": 769, "p": 9, "k": 162},
        # supervised segmentation of a data term: 5 labels, no label cost
        {"name": "segment_5_481x321", "kind": "segment", "W": 481, "H": 321, "n_labels": 5,
         "lam": 4.0, "nu": 0.0, "iterations": 300},
        # unsupervised segmentation: 16 segments with the MDL label cost
        {"name": "segment_mdl_16_481x321", "kind": "segment", "W": 481, "H": 321, "n_labels": 16,
         "lam": 6.0, "nu": 1100.0, "iterations": 300},
        # its data term: k-means and k-medians, 4 x 4 classes, 10 rounds each
        {"name": "unsup_4x4_481x321", "kind": "unsup", "W": 481, "H": 321, "nc": 4, "nt": 4,
         "p": 7, "k": 98, "rounds": 10},
        # a planned batch of uneven images, refilled and run again (serving)
        {"name": "batch_fp8_12", "kind": "batch", "images": 12, "shapes": 7, "p": 7, "k": 98,
         "precision": "fp8"},
        # forward and backward of the surrogate's network: one training step of
        # 152 x 128 rows, extended features of 10 labels
        {"name": "mlp_grad_19456", "kind": "mlp_grad", "rows": 19456, "n_in": 55, "n_out": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["data_term"] * 5 + ["codes", "segment", "segment", "unsup", "batch",
                                           "mlp_grad"])
    if kind == "data_term":
        precision = rng.choice(["fp32", "bf16", "fp8", "fp8"])
        p = rng.choice([3, 5, 7, 7] if precision == "bf16" else [5, 7, 7, 9])
        W, H, n = _log(rng, 64, 1024), _log(rng, 48, 1024), rng.randint(2, 10)
        most = {"fp32": 1.5e10, "bf16": 4e10, "fp8": 8e10}[precision]  # pixel x sample pairs
        m = min(_log(rng, 60, 20000), max(20, int(most / (W * H * n))))
        return {"kind": kind, "W": W, "H": H, "n_labels": n, "m": m, "p": p, "k": 2 * p * p,
                "precision": precision,
                "mode": rng.choice(["persample", "persample", "factorised", "smooth"]),
                "all_outputs": rng.random() < 0.5, "uneven": rng.random() < 0.5}
    if kind == "codes":
        p = rng.choice([3, 5, 7, 9])
        return {"kind": kind, "W": _log(rng, 64, 2048), "H": _log(rng, 48, 1536), "p": p,
                "k": 2 * p * p}
    if kind == "segment":
        return {"kind": kind, "W": _log(rng, 64, 640), "H": _log(rng, 48, 480),
                "n_labels": rng.randint(2, 16), "lam": rng.choice([2.0, 4.0, 6.0, 8.0]),
                "nu": rng.choice([0.0, 0.0, 50.0, 1100.0]), "iterations": rng.randint(100, 300)}
    if kind == "unsup":
        p = rng.choice([5, 7, 9])
        return {"kind": kind, "W": _log(rng, 96, 640), "H": _log(rng, 64, 480),
                "nc": rng.randint(2, 6), "nt": rng.randint(2, 6), "p": p, "k": 2 * p * p,
                "rounds": rng.randint(4, 10)}
    if kind == "batch":
        return {"kind": kind, "images": rng.randint(3, 12), "shapes": rng.randint(0, 10 ** 6),
                "p": 7, "k": 98, "precision": rng.choice(["fp8", "fp8", "bf16"])}
    n = rng.randint(2, 19)
    return {"kind": kind, "rows": _log(rng, 256, 32768), "n_in": rng.choice([21, 45 + n]),
            "n_out": n}


# ------------------------------------------------------------------ inputs


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _u(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device=DEV)


def _regions(g, W, H, n):
    """Voronoi cells (H, W) of n sites on a jittered grid, so that no cell is tiny."""
    cols = max(1, round(math.sqrt(n * W / H)))
    rows = -(-n // cols)
    cell = torch.randperm(rows * cols, generator=g, device=DEV)[:n]
    sx = ((cell % cols) + _u(g, 0.25, 0.75, n)) * (W / cols)
    sy = (torch.div(cell, cols, rounding_mode="floor") + _u(g, 0.25, 0.75, n)) * (H / rows)
    x = torch.arange(W, device=DEV, dtype=torch.float32)
    y = torch.arange(H, device=DEV, dtype=torch.float32)
    best = torch.full((H, W), math.inf, device=DEV)
    reg = torch.zeros((H, W), dtype=torch.int64, device=DEV)
    for r in range(n):
        d = (x[None, :] - sx[r]) ** 2 + (y[:, None] - sy[r]) ** 2
        near = d < best
        best = torch.where(near, d, best)
        reg[near] = r
    return reg


def _image(g, reg, n):
    """Gratings (even cells) and checkerboards (odd cells) times a tint, plus noise."""
    H, W = reg.shape
    period, theta = _u(g, 3.0, 12.0, n)[reg], _u(g, 0.0, math.pi, n)[reg]
    phase, tint = _u(g, 0.0, 2 * math.pi, n)[reg], _u(g, 0.2, 1.0, n, 3)[reg]
    x = torch.arange(W, device=DEV, dtype=torch.float32)[None, :]
    y = torch.arange(H, device=DEV, dtype=torch.float32)[:, None]
    u = torch.cos(theta) * x + torch.sin(theta) * y
    v = -torch.sin(theta) * x + torch.cos(theta) * y
    check = (torch.floor(u / period + phase / (2 * math.pi)) + torch.floor(v / period)) % 2
    wave = 0.5 + 0.5 * torch.sin(2 * math.pi * u / period + phase)
    val = torch.where(reg % 2 == 1, 0.15 + 0.7 * check, wave)
    img = val[..., None] * tint + 0.05 * torch.randn((H, W, 3), generator=g, device=DEV)
    return img.clamp(0.0, 1.0).contiguous()


def _scribble(g, reg, label, want):
    """Unique pixels of one cell from random-walk strokes, in random order."""
    H, W = reg.shape
    inside = reg.reshape(-1) == label
    cand = torch.nonzero(inside).flatten()
    want = max(1, min(want, cand.numel() // 2))
    got = cand[:0]
    strokes = 16 + want // 8
    dy = torch.tensor([0, 0, 1, 1, -1, 0, 1, -1, -1], device=DEV)
    dx = torch.tensor([0, 1, 0, 1, -1, -1, -1, 0, 1], device=DEV)
    size = torch.tensor([1, 4, 9], device=DEV)  # brushes of 1, 2 x 2 and 3 x 3 pixels
    for _ in range(12):
        s = cand[torch.randint(cand.numel(), (strokes,), generator=g, device=DEV)]
        head = _u(g, 0.0, 2 * math.pi, strokes)[:, None] + torch.cumsum(
            0.3 * torch.randn((strokes, 60), generator=g, device=DEV), 1)
        x = torch.round((s % W)[:, None] + torch.cumsum(torch.cos(head), 1)).long()
        y = torch.round(torch.div(s, W, rounding_mode="floor")[:, None]
                        + torch.cumsum(torch.sin(head), 1)).long()
        length = torch.randint(15, 61, (strokes,), generator=g, device=DEV)
        on = torch.arange(60, device=DEV)[None, :] < length[:, None]
        on &= (x >= 0) & (x < W) & (y >= 0) & (y < H)
        on &= inside[(y.clamp(0, H - 1) * W + x.clamp(0, W - 1))]
        on = torch.cumprod(on.to(torch.int32), 1).bool()  # a stroke ends where it leaves the cell
        brush = size[torch.randint(3, (strokes,), generator=g, device=DEV)]
        bx, by = x[..., None] + dx, y[..., None] + dy
        ok = on[..., None] & (torch.arange(9, device=DEV) < brush[:, None])[:, None, :]
        ok &= (bx >= 0) & (bx < W) & (by >= 0) & (by < H)
        pix = (by * W + bx)[ok]
        got = torch.unique(torch.cat([got, pix[inside[pix]]]))
        if got.numel() >= want:
            break
        strokes *= 2
    if got.numel() < want:
        got = torch.unique(torch.cat([got, cand]))
    return got[torch.randperm(got.numel(), generator=g, device=DEV)[:want]].to(torch.int32)


def _operator(g, p, k):
    om = torch.randn((k, p * p), generator=g, device=DEV, dtype=torch.float64)
    om = (om / om.norm(dim=1, keepdim=True)).float().contiguous()
    r = torch.arange(p, device=DEV, dtype=torch.float64) - (p - 1) / 2
    w = torch.exp(-(r[:, None] ** 2 + r[None, :] ** 2) / (2.0 * (p / 4.0) ** 2))
    return om, w.reshape(-1).float().contiguous()


def _scene(g, W, H, counts):
    """An image and its scribbles: counts[i] samples wanted of label i, one cell more than labels."""
    n = len(counts)
    reg = _regions(g, W, H, n + 1)
    img = _image(g, reg, n + 1)
    pix = []
    for i, m in enumerate(counts):
        if not bool((reg == i).any()):  # a cell that no pixel is nearest to
            reg[0, i] = i
        pix.append(_scribble(g, reg, i, m))
    off = np.zeros(n + 1, np.int32)
    off[1:] = np.cumsum([t.numel() for t in pix])
    return {"img": img, "label_off": off, "sample_pix": torch.cat(pix).contiguous()}


def _counts(case):
    n, m = case["n_labels"], case["m"]
    if not case.get("uneven"):
        return [m] * n
    return [max(1, m * (i + 1) ** 2 // n ** 2) for i in range(n)]  # the last label has m


def _batch_shapes(case):
    """(W, H, samples per label) of every image: the batch workload's recipe."""
    r = random.Random(case["shapes"])
    return [(r.randint(240, 640), r.randint(160, 480),
             [r.randint(500, 5000) for _ in range(r.randint(2, 10))])
            for _ in range(case["images"])]


def _inputs(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    d = {}
    if kind == "data_term":
        d = _scene(g, case["W"], case["H"], _counts(case))
    elif kind == "batch":
        d["images"] = [_scene(g, W, H, m) for W, H, m in _batch_shapes(case)]
    elif kind in ("codes", "unsup"):
        d["img"] = _image(g, _regions(g, case["W"], case["H"], 6), 6)
    elif kind == "segment":
        # a data term as the likelihoods give it: around 8 nats, the right
        # label a nat or so lower over its cell, noisy from pixel to pixel
        n = case["n_labels"]
        reg = _regions(g, case["W"], case["H"], n)
        d["img"] = _image(g, reg, n)
        f = 8.0 + 0.5 * torch.randn((n, case["H"], case["W"]), generator=g, device=DEV)
        f += _u(g, 0.6, 1.6, n)[:, None, None] * (reg[None] != torch.arange(n, device=DEV)[:, None,
                                                                                         None])
        d["f"] = f.contiguous()
    elif kind == "mlp_grad":
        nin, n = case["n_in"], case["n_out"]
        w = []
        for rows, cols in ((64, nin), (64, 64), (64, 64), (n, 64)):
            w += [torch.randn((rows, cols), generator=g, device=DEV) * math.sqrt(2.0 / cols),
                  0.1 * torch.randn((rows,), generator=g, device=DEV)]
        d["params"] = torch.cat([t.reshape(-1) for t in w]).contiguous()
        d["X"] = torch.randn((case["rows"], nin), generator=g, device=DEV)
        d["T"] = torch.randn((case["rows"], n), generator=g, device=DEV)
    if "p" in case:
        d["omega"], d["mask"] = _operator(g, case["p"], case["k"])
    if kind == "unsup":
        P = case["W"] * case["H"]
        r = np.random.default_rng(seed)
        d["ci"] = r.choice(P, case["nc"], replace=False).astype(np.int32)
        d["ti"] = r.choice(P, case["nt"], replace=False).astype(np.int32)
    return d


def prepare(case, seed):
    """The inputs, the context, the outputs' buffers (a program keeps them and
    refills the inputs) and, for a batch, its plan."""
    kind = case["kind"]
    s = _inputs(case, seed)
    s["kind"], s["ctx"] = kind, context()
    if kind == "data_term":
        n, H, W, k = case["n_labels"], case["H"], case["W"], case["k"]
        s["prm"] = cs.Params.default(p=case["p"], mode=MODE[case["mode"]],
                                     precision=PRECISION[case["precision"]])
        s["out"] = {"neglog": torch.empty((n, H, W), device=DEV),
                    "post": torch.empty((n, H, W), device=DEV), "dist2": None, "bitmask": None}
        if case["all_outputs"]:
            s["out"]["dist2"] = torch.empty((n, H, W), dtype=torch.int32, device=DEV)
            s["out"]["bitmask"] = torch.empty((H * W, (k + 31) // 32), dtype=torch.int32,
                                              device=DEV)
    elif kind == "codes":
        s["prm"] = cs.Params.default(p=case["p"])
    elif kind == "segment":
        s["sp"] = cs.SegParams.default(lam=case["lam"], nu=case["nu"],
                                       iterations=case["iterations"])
        n, H, W = s["f"].shape
        s["out"] = {"u": torch.empty((n, H, W), device=DEV),
                    "labels": torch.empty((H, W), dtype=torch.int32, device=DEV)}
    elif kind == "unsup":
        s["prm"] = cs.Params.default(p=case["p"], sigma_c2=UNSUP_SIGMA_C2)
        s["up"] = cs.UnsupParams.default(n_colour=case["nc"], n_texture=case["nt"],
                                         kmeans_iterations=case["rounds"],
                                         kmedians_iterations=case["rounds"], beta=UNSUP_BETA)
    elif kind == "batch":
        s["prm"] = cs.Params.default(p=case["p"], precision=PRECISION[case["precision"]])
        s["batch"] = s["ctx"].batch(s["images"], s["omega"], s["mask"], s["prm"],
                                    flags=cs.BATCH_GRAPH)
    return s


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "data_term":
        return ctx.data_term(s["img"], s["omega"], s["mask"], s["label_off"], s["sample_pix"],
                             s["prm"], out=s["out"])
    if kind == "codes":
        out = ctx.codes(s["img"], s["omega"], s["mask"], s["prm"], want_lead16=True)
        return {"bitmask": out["bitmask"], "lead16": out["lead16"]}
    if kind == "segment":
        return ctx.segment(s["f"], s["img"], s["sp"], out=s["out"])
    if kind == "unsup":
        return ctx.unsup_data_term(s["img"], s["omega"], s["mask"], s["prm"], s["up"], s["ci"],
                                   s["ti"])
    if kind == "batch":
        return [{"neglog": o["neglog"], "post": o["post"]} for o in s["batch"].run()]
    return ctx.mlp_grad(s["params"], s["T"].shape[1], s["X"], s["T"])


# ------------------------------------------------------------------ work


def _likelihood_work(W, H, n, S, p, k, texture):
    P = W * H
    # per pair: the co-support product, the location and colour distances, the
    # exponent, the exponential and the sum; per pixel: the patch and its codes
    flops = P * S * ((2 * k if texture else 0) + 21) + P * (2 * k * p * p + 8 * p * p)
    return 4 * (3 * P + k * p * p + p * p + S + 2 * n * P), flops


def work(case):
    kind = case["kind"]
    if kind == "data_term":
        W, H, n, k, p = (case[c] for c in ("W", "H", "n_labels", "k", "p"))
        b, f = _likelihood_work(W, H, n, sum(_counts(case)), p, k, case["mode"] == "persample")
        if case["all_outputs"]:
            b += 4 * W * H * (n + (k + 31) // 32)
        if case["mode"] != "persample":
            f += 3 * W * H * n * k
        return {"bytes": b, "flops": f}
    if kind == "codes":
        P, k, n = case["W"] * case["H"], case["k"], case["p"] ** 2
        return {"bytes": 4 * (3 * P + k * n + n + P * ((k + 31) // 32 + 16)),
                "flops": P * (2 * k * n + 8 * n)}
    if kind == "segment":
        P, n = case["W"] * case["H"], case["n_labels"]
        return {"bytes": 4 * P * (2 * n + 3 + 1), "flops": case["iterations"] * P * n * 40}
    if kind == "unsup":
        P, k, n = case["W"] * case["H"], case["k"], case["p"] ** 2
        nc, nt, r = case["nc"], case["nt"], case["rounds"]
        return {"bytes": 4 * P * (3 + nc * nt + 2),
                "flops": P * (2 * k * n + (r + 1) * (8 * nc + 2 * k * nt) + r * 4 * k)}
    if kind == "batch":
        w = [_likelihood_work(W, H, len(m), sum(m), case["p"], case["k"], True)
             for W, H, m in _batch_shapes(case)]
        return {"bytes": sum(b for b, _ in w), "flops": sum(f for _, f in w)}
    nin, n, B = case["n_in"], case["n_out"], case["rows"]
    np_ = 64 * nin + 2 * 64 * 64 + 3 * 64 + 64 * n + n
    return {"bytes": 4 * (B * (nin + n) + 2 * np_), "flops": 6 * B * np_}


# ------------------------------------------------------------------ float64 restatement


def _patches(img, p, mask):
    """Normalised masked patches (P, p p) in float64: window clamped at the edge."""
    x = img.double()
    gray = 0.299 * x[..., 0] + 0.587 * x[..., 1] + 0.114 * x[..., 2]
    r = (p - 1) // 2
    H, W = gray.shape
    yy = torch.arange(-r, H + r, device=DEV).clamp(0, H - 1)
    xx = torch.arange(-r, W + r, device=DEV).clamp(0, W - 1)
    pad = gray[yy][:, xx]
    v = pad.unfold(0, p, 1).unfold(1, p, 1).reshape(H * W, p * p) * mask.double()
    v = v - v.mean(1, keepdim=True)
    nrm = v.norm(dim=1, keepdim=True)
    return torch.where(nrm > 1e-13, v / nrm.clamp_min(1e-300), torch.zeros_like(v))


def _codes(d, p):
    return _patches(d["img"], p, d["mask"]) @ d["omega"].double().T


def _median_rows(v):
    """Column medians of v (m, k): the mean of the two middle values for an even count."""
    s, m = torch.sort(v, 0).values, v.shape[0]
    return 0.5 * (s[(m - 1) // 2] + s[m // 2])


def _data_term(d, p, mode):
    img = d["img"].double()
    H, W, _ = img.shape
    P = H * W
    off, smp = d["label_off"], d["sample_pix"].long()
    n = len(off) - 1
    col = img.reshape(P, 3)
    q = torch.arange(P, device=DEV)
    px, py = (q % W).double(), torch.div(q, W, rounding_mode="floor").double()
    a = _codes(d, p)
    bits = (a.abs() <= TAU).float()
    pop = bits.sum(1)
    L = torch.empty((n, P), dtype=torch.float64, device=DEV)
    beta = torch.empty_like(L)
    for i in range(n):
        s = smp[int(off[i]):int(off[i + 1])]
        step = max(1, 40_000_000 // s.numel())
        for lo in range(0, P, step):
            e = slice(lo, min(P, lo + step))
            d2 = (px[e, None] - px[s]) ** 2
            d2 += (py[e, None] - py[s]) ** 2
            rho = ALPHA * d2.min(1, keepdim=True).values.sqrt().clamp_min(D_MIN)
            beta[i, e] = KAPPA * rho[:, 0]
            d2 *= -0.5 / rho ** 2
            c2 = (col[e, None, 0] - col[s, 0]) ** 2
            for c in (1, 2):
                c2 += (col[e, None, c] - col[s, c]) ** 2
            d2 -= c2 * (0.5 / SIGMA_C2)
            del c2
            if mode == "persample":
                ham = pop[e, None] + pop[s] - 2.0 * (bits[e] @ bits[s].T)
                d2 -= ham.double() / beta[i, e, None]
            L[i, e] = (torch.logsumexp(d2, 1) - math.log(s.numel())
                       - torch.log(2 * math.pi * rho[:, 0] ** 2)
                       - 1.5 * math.log(2 * math.pi * SIGMA_C2))
    if mode != "persample":
        t = torch.empty_like(L)
        iota = torch.exp(-a * a / IOTA_SIGMA) if mode == "smooth" else bits.double()
        for i in range(n):
            v = iota[smp[int(off[i]):int(off[i + 1])]]
            rep = _median_rows(v) if mode == "smooth" else (2 * v.sum(0) >= v.shape[0]).double()
            t[i] = -(iota - rep).abs().sum(1) / beta[i]
        L += torch.log_softmax(t, 0)
    return {"neglog": -L.reshape(n, H, W), "post": torch.softmax(L, 0).reshape(n, H, W),
            "dist2": None, "bitmask": None}


def _segment(f, img, lam, nu, iterations, gamma=5.0):
    f, I = f.double(), 255.0 * img.double().permute(2, 0, 1)
    n, H, W = f.shape

    def grad(v):
        gx, gy = torch.zeros_like(v), torch.zeros_like(v)
        gx[..., :, :-1] = v[..., :, 1:] - v[..., :, :-1]
        gy[..., :-1, :] = v[..., 1:, :] - v[..., :-1, :]
        return gx, gy

    gx, gy = grad(I)
    bound = 0.5 * lam * torch.exp(-(gx * gx + gy * gy).sum(0).sqrt() / gamma) / (2 * gamma)
    u = torch.full_like(f, 1.0 / n)
    ub, px, py, mu = u.clone(), torch.zeros_like(f), torch.zeros_like(f), torch.zeros_like(f)
    m, mb = torch.ones(n, dtype=torch.float64, device=DEV), torch.ones(n, dtype=torch.float64,
                                                                       device=DEV)
    rank = torch.arange(1, n + 1, device=DEV, dtype=torch.float64)[:, None, None]
    for _ in range(iterations):
        gx, gy = grad(ub)
        px += 0.5 * gx
        py += 0.5 * gy
        sc = (torch.sqrt(px * px + py * py) / bound.clamp_min(1e-300)).clamp_min(1.0)
        px /= sc
        py /= sc
        mu = (mu + 0.5 * (mb[:, None, None] - ub)).clamp_max(0.0)
        mn = (m - (nu + mu.sum((1, 2))) / (H * W)).clamp(0.0, 1.0)
        mb, m = 2 * mn - m, mn
        qx, qy = px.clone(), py.clone()  # div: no flux across the last column and row
        qx[..., :, -1] = 0
        qy[..., -1, :] = 0
        div = qx + qy
        div[..., :, 1:] -= qx[..., :, :-1]
        div[..., 1:, :] -= qy[..., :-1, :]
        v = u - 0.2 * (f - div - mu)
        s = torch.sort(v, 0, descending=True).values  # projection onto the simplex
        c = (torch.cumsum(s, 0) - 1.0) / rank
        k = ((s > c).sum(0, keepdim=True) - 1).clamp_min(0)
        un = (v - torch.gather(c, 0, k)).clamp_min(0.0)
        ub, u = 2 * un - u, un
    return {"u": u, "labels": None}


def _unsup(d, case):
    img = d["img"].double()
    H, W, _ = img.shape
    P, nc, nt = H * W, case["nc"], case["nt"]
    X = img.reshape(P, 3)
    V = torch.exp(-_codes(d, case["p"]) ** 2 / IOTA_SIGMA)  # (P, k)

    def far(points, C, power):
        return torch.stack([(points - c).abs().pow(power).sum(1) for c in C])

    def clusters(points, start, power, centre):
        C = points[torch.as_tensor(start, device=DEV).long()].clone()
        for _ in range(case["rounds"]):
            lab = torch.argmin(far(points, C, power), 0)
            C = torch.stack([centre(points[lab == i]) if bool((lab == i).any()) else C[i]
                             for i in range(len(C))])
        return C

    cc = clusters(X, d["ci"], 2, lambda v: v.mean(0))
    tc = clusters(V, d["ti"], 1, _median_rows)
    lc = torch.log_softmax(-far(X, cc, 2) / (2 * UNSUP_SIGMA_C2), 0)
    lt = torch.log_softmax(-far(V, tc, 1) / UNSUP_BETA, 0)
    f = -(lc[:, None] + lt[None]).reshape(nc * nt, H, W)
    return {"neglog": f, "colour_centres": cc, "texture_centres": tc, "colour_assign": None,
            "texture_assign": None}


def _mlp_grad(d, nin, n):
    p = d["params"].bfloat16().double()  # the network's weights are used rounded to bf16
    w, o = [], 0
    for shape in ((64, nin), (64,), (64, 64), (64,), (64, 64), (64,), (n, 64), (n,)):
        size = math.prod(shape)
        w.append(p[o:o + size].reshape(shape).requires_grad_(True))
        o += size
    h = d["X"].double()
    for layer in range(3):
        h = torch.nn.functional.silu(h @ w[2 * layer].T + w[2 * layer + 1])
    z = h @ w[6].T + w[7]
    loss = 0.5 * ((z - d["T"].double()) ** 2).mean()
    grads = torch.autograd.grad(loss, w)
    return torch.cat([t.reshape(-1) for t in grads]), loss.detach().reshape(1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "data_term" and case["W"] * case["H"] * sum(_counts(case)) > 4e10:
        return None  # over 20 seconds in float64
    if kind == "batch" and sum(W * H * sum(m) for W, H, m in _batch_shapes(case)) > 4e10:
        return None
    d = _inputs(case, seed)
    if kind == "data_term":
        return _data_term(d, case["p"], case["mode"])
    if kind == "codes":
        a = _codes(d, case["p"])[:, :16]
        return {"bitmask": None, "lead16": torch.nn.functional.pad(a, (0, 16 - a.shape[1]))}
    if kind == "segment":
        return _segment(d["f"], d["img"], case["lam"], case["nu"], case["iterations"])
    if kind == "unsup":
        return _unsup(d, case)
    if kind == "batch":
        out = []
        for m in d["images"]:
            o = _data_term(dict(m, omega=d["omega"], mask=d["mask"]), case["p"], "persample")
            out.append({"neglog": o["neglog"], "post": o["post"]})
        return out
    return _mlp_grad(d, case["n_in"], case["n_out"])
