"""Workloads a user of libms runs, for timing one version of the library against another.

Every case goes through the Python binding's public calls. Frames follow the
repository's own synthetic recipes (von Mises-Fisher cells laid out like
microscopy frames, 2% outliers, norms in [0.5, 2]; the 18-d orthogonal blobs
of the simulation suite; unit pixels of many cells for the smooth kernel),
drawn on the GPU so that making them is quick.
"""
import math

import numpy as np
import torch

import paper_2007_14283_gb300 as ms
from paper_2007_14283_gb300.autograd import vmf_mean_shift

DEV = "cuda"
#: Seed-iterations per foreground pixel of a frame of vMF cells with kappa in
#: [20, 200] at bandwidth 0.9: 310,102 on a 512 x 512 frame of 131,072 pixels.
SEED_ITERS_PER_PIXEL = 2.37


def listed():
    return [
        # One small field of view, the shortest call: every pixel foreground, library defaults (FP32).
        dict(name="frame_64", kind="frame", H=64, W=64, d=16, fill=1.0, cells=8, kappa_lo=50.0, kappa_hi=50.0,
             outliers=0.0, precision="fp32", bandwidth=0.9, n_initial=128),
        # The simulation design: 18-d blobs, well separated, so one or two rounds and few modes.
        dict(name="blobs_20k", kind="blobs", n=20011, d=18, clusters=10, precision="fp32", bandwidth=0.9, n_initial=128),
        # A camera frame with its background masked, library defaults (FP32).
        dict(name="frame_512_fp32", kind="frame", H=512, W=512, d=16, fill=0.5, cells=60, kappa_lo=20.0, kappa_hi=200.0,
             outliers=0.02, precision="fp32", bandwidth=0.9, n_initial=128),
        # The same in the BF16 tensor-core form, the usual choice for throughput.
        dict(name="frame_512_bf16", kind="frame", H=512, W=512, d=16, fill=0.5, cells=60, kappa_lo=20.0, kappa_hi=200.0,
             outliers=0.02, precision="bf16", bandwidth=0.9, n_initial=128),
        # A network with a wider embedding on a frame of odd size.
        dict(name="frame_481x519_d24", kind="frame", H=481, W=519, d=24, fill=0.5, cells=60, kappa_lo=20.0, kappa_hi=200.0,
             outliers=0.02, precision="bf16", bandwidth=0.9, n_initial=128),
        # Serving: frames of uneven size in one graph launch, the batch object kept between calls.
        dict(name="batch_24_uneven", kind="batch", frames=24, n_lo=2000, n_hi=200000, d=16, precision="bf16", bandwidth=0.9),
        # Serving many small crops.
        dict(name="batch_30_small", kind="batch", frames=30, n_lo=300, n_hi=4000, d=16, precision="bf16", bandwidth=0.9),
        # A cell-tracking sequence: consecutive frames whose cells drift, N carried from frame to frame.
        dict(name="video_4x512", kind="video", frames=4, H=512, W=512, d=16, fill=0.5, cells=60, precision="bf16",
             bandwidth=0.9),
        # A frame that starts and ends in host memory (a camera process without a GPU pipeline).
        dict(name="host_257x250", kind="host", H=257, W=250, d=16, fill=0.5, cells=30, kappa_lo=20.0, kappa_hi=200.0,
             outliers=0.02, precision="bf16", bandwidth=0.9, n_initial=128),
        # Training through the smooth kernel, FP32: forward and backward of ten unrolled steps.
        dict(name="train_fp32", kind="train", N=65536, M=1024, T=10, kappa=20.0, precision="fp32"),
        # The same on the tensor cores, at an odd size.
        dict(name="train_bf16", kind="train", N=50021, M=900, T=8, kappa=20.0, precision="bf16"),
        # Dense mean-shift with another distance and profile.
        dict(name="shift_gauss", kind="kshift", N=65536, M=1024, d=16, T=10, distance="euclid", profile="gaussian", h=0.45),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "blobs", "batch", "video", "host", "train", "kshift"])
    precision = rng.choice(["fp32", "bf16"])
    bandwidth = rng.choice([0.87, 0.9, 0.9, 0.93])
    if kind in ("frame", "host"):
        d = rng.choice([8, 16, 16, 16, 17, 24, 32])
        fill = rng.choice([0.3, 0.5, 0.8, 1.0])
        top = 60000 if d > 16 and precision == "fp32" else 130000
        area = _log(rng, 1500, int(top / fill))
        W = max(16, int(math.sqrt(area) * rng.uniform(0.7, 1.4)))
        H = max(16, area // W)
        lo = rng.choice([20.0, 20.0, 50.0, 100.0])
        return dict(kind=kind, H=H, W=W, d=d, fill=fill, cells=max(3, min(120, int(H * W * fill / rng.uniform(400, 3000)))),
                    kappa_lo=lo, kappa_hi=200.0, outliers=0.02 if fill < 1.0 else 0.0, precision=precision,
                    bandwidth=bandwidth, n_initial=rng.choice([64, 128, 256]))
    if kind == "blobs":
        d = rng.choice([12, 18, 18, 31])
        return dict(kind=kind, n=_log(rng, 1000, 200000), d=d, clusters=10, precision=precision, bandwidth=0.9,
                    n_initial=rng.choice([64, 128, 256]))
    if kind == "batch":
        hi = _log(rng, 2000, 60000 if precision == "fp32" else 150000)
        return dict(kind=kind, frames=rng.randint(2, 20), n_lo=max(200, hi // rng.choice([4, 16, 64])), n_hi=hi,
                    d=16 if precision == "fp32" else rng.choice([16, 16, 32]), precision=precision, bandwidth=bandwidth)
    if kind == "video":
        side = _log(rng, 96, 512 if precision == "bf16" else 330)
        return dict(kind=kind, frames=rng.randint(2, 4), H=side, W=side + rng.randint(-9, 9), d=16, fill=0.5,
                    cells=max(3, side * side // 4400), precision=precision, bandwidth=bandwidth)
    if kind == "train":
        return dict(kind=kind, N=_log(rng, 700, 90000), M=_log(rng, 40, 1100), T=rng.randint(1, 10),
                    kappa=rng.choice([5.0, 10.0, 20.0, 40.0]), precision=precision)
    distance = rng.choice(["cosine", "euclid"])
    return dict(kind=kind, N=_log(rng, 700, 90000), M=_log(rng, 40, 1100), d=rng.choice([8, 16, 16, 18, 32]),
                T=rng.randint(1, 10), distance=distance, profile=rng.choice(["flat", "epanechnikov", "gaussian"]),
                h=0.1 if distance == "cosine" else 0.45)


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)


def _sphere(g, n, d):
    v = torch.randn(n, d, generator=g, device=DEV, dtype=torch.float64)
    return v / v.norm(dim=1, keepdim=True)


def _vmf(g, means, kappas, owner):
    """One vMF(means[k], kappas[k]) sample per entry of owner (float64 [n, d]): the cosine to the mean from
    its inverse distribution function on a grid, a uniform direction in the tangent space."""
    K, d = means.shape
    n = owner.numel()
    w = torch.linspace(-1.0, 1.0, 4097, device=DEV, dtype=torch.float64)[1:-1]
    logp = kappas[:, None] * (w - 1.0) + 0.5 * (d - 3) * torch.log1p(-w * w)
    cdf = torch.cumsum(torch.exp(logp - logp.max(dim=1, keepdim=True).values), dim=1)
    cdf = cdf / cdf[:, -1:]
    flat = (cdf + torch.arange(K, device=DEV, dtype=torch.float64)[:, None]).reshape(-1)
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    at = torch.searchsorted(flat, u + owner).clamp_(max=flat.numel() - 1) - owner * w.numel()
    at = at.clamp_(0, w.numel() - 1)
    step = 2.0 / 4096
    cw = (w[at] + (torch.rand(n, generator=g, device=DEV, dtype=torch.float64) - 0.5) * step).clamp_(-1.0, 1.0)
    mu = means[owner]
    v = torch.randn(n, d, generator=g, device=DEV, dtype=torch.float64)
    v -= (v * mu).sum(1, keepdim=True) * mu
    v /= v.norm(dim=1, keepdim=True)
    return cw[:, None] * mu + torch.sqrt((1.0 - cw * cw).clamp_(min=0.0))[:, None] * v


def _layout(g, H, W, n_cell, cells):
    """Cell index of every pixel (-1 outside): elliptical blobs around random centres, n_cell pixels in all."""
    y = torch.arange(H, device=DEV, dtype=torch.float32).repeat_interleave(W)
    x = torch.arange(W, device=DEV, dtype=torch.float32).repeat(H)
    r = torch.rand(cells, 4, generator=g, device=DEV)
    size = torch.exp(0.37 * torch.randn(cells, generator=g, device=DEV))
    best = torch.full((H * W,), math.inf, device=DEV)
    owner = torch.zeros(H * W, dtype=torch.int64, device=DEV)
    ct, st = torch.cos(math.pi * r[:, 2]), torch.sin(math.pi * r[:, 2])
    aspect = 1.0 + 0.6 * r[:, 3]
    for k in range(cells):
        dy, dx = y - r[k, 0] * H, x - r[k, 1] * W
        a, b = dx * ct[k] + dy * st[k], dy * ct[k] - dx * st[k]
        m = (a * a / aspect[k] + b * b * aspect[k]) / size[k]
        closer = m < best
        best = torch.where(closer, m, best)
        owner = torch.where(closer, torch.full_like(owner, k), owner)
    if n_cell < H * W:
        owner[torch.argsort(best, stable=True)[n_cell:]] = -1
    return owner


def _frame(g, H, W, d, fill, cells, kappa_lo, kappa_hi, outliers, means=None, kappas=None, owner=None):
    n_fg = max(1, int(round(fill * H * W)))
    n_out = int(outliers * n_fg)
    if owner is None:
        owner = _layout(g, H, W, n_fg - n_out, cells)
    if means is None:
        means = _sphere(g, cells, d)
    if kappas is None:
        kappas = kappa_lo + (kappa_hi - kappa_lo) * torch.rand(cells, generator=g, device=DEV, dtype=torch.float64)
    fg = owner >= 0
    emb = torch.randn(H * W, d, generator=g, device=DEV, dtype=torch.float64)
    scale = 0.5 + 1.5 * torch.rand(H * W, generator=g, device=DEV, dtype=torch.float64)
    idx = torch.nonzero(fg).reshape(-1)
    emb[idx] = _vmf(g, means, kappas, owner[idx])
    mask = None
    if n_fg < H * W:
        free = torch.nonzero(~fg).reshape(-1)
        pick = free[torch.randperm(free.numel(), generator=g, device=DEV)[:n_out]]
        emb[pick] = _sphere(g, pick.numel(), d)
        fg[pick] = True
        mask = fg.to(torch.uint8)
    return (emb * scale[:, None]).float().contiguous(), mask


def _blobs(g, n, d, clusters):
    centre = torch.zeros(clusters, d, device=DEV, dtype=torch.float64)
    for k in range(clusters):
        centre[k, k // 2] = 1.0 if k % 2 == 0 else -1.0
    truth = (torch.arange(n, device=DEV) % clusters)[torch.randperm(n, generator=g, device=DEV)]
    return (centre[truth] + 0.01 * torch.randn(n, d, generator=g, device=DEV, dtype=torch.float64)).float().contiguous()


def _points(g, N, M, d):
    """N unit vectors of 32 vMF cells, M of them as seeds, and each seed's cell mean."""
    means = _sphere(g, 32, d)
    kappas = 20.0 + 180.0 * torch.rand(32, generator=g, device=DEV, dtype=torch.float64)
    owner = torch.randint(0, 32, (N,), generator=g, device=DEV)
    P = _vmf(g, means, kappas, owner)
    at = torch.randperm(N, generator=g, device=DEV)[torch.arange(M, device=DEV) % N]
    return P.float().contiguous(), P[at].float().contiguous(), means[owner[at]].float().contiguous()


def _batch_sizes(case):
    lo, hi, B = case["n_lo"], case["n_hi"], case["frames"]
    return [int(round(lo * (hi / lo) ** ((i + 0.5) / B))) for i in range(B)]


def _precision(case):
    return ms.MS_BF16 if case["precision"] == "bf16" else ms.MS_FP32


def _options(case):
    o = dict(precision=_precision(case), bandwidth_cos=case["bandwidth"], merge_cos=case["bandwidth"])
    if "n_initial" in case:
        o["n_initial"] = case["n_initial"]
    return o


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("frame", "host"):
        emb, mask = _frame(g, case["H"], case["W"], case["d"], case["fill"], case["cells"], case["kappa_lo"],
                           case["kappa_hi"], case["outliers"])
        n_fg = emb.shape[0] if mask is None else int(mask.sum().item())
        s.update(emb=emb, mask=mask, cfg=ms.ms_config_default(dim=case["d"], **_options(case)),
                 labels=torch.empty(emb.shape[0], dtype=torch.int32, device=DEV),
                 modes=torch.zeros(n_fg, emb.shape[1], dtype=torch.float32, device=DEV))
        if kind == "host":
            for key in ("emb", "mask", "labels", "modes"):
                s[key] = None if s[key] is None else s[key].cpu().pin_memory()
    elif kind == "blobs":
        s.update(emb=_blobs(g, case["n"], case["d"], case["clusters"]), mask=None)
    elif kind == "batch":
        embs, masks = [], []
        for n in _batch_sizes(case):
            side = max(16, int(math.ceil(math.sqrt(2 * n))))
            cells = int(torch.randint(5, 121, (1,), generator=g, device=DEV).item())
            e, m = _frame(g, side, side, case["d"], n / (side * side), max(1, min(cells, n // 40)), 20.0, 200.0, 0.02)
            embs.append(e)
            masks.append(m)
        s["modes"] = [np.zeros((n, case["d"]), dtype=np.float32) for n in _batch_sizes(case)]
        s["batch"] = ms.ms_batch_create(ms.ms_config_default(dim=case["d"], **_options(case)), embs, masks)
    elif kind == "video":
        H, W, d, cells = case["H"], case["W"], case["d"], case["cells"]
        n_fg = int(round(case["fill"] * H * W))
        owner = _layout(g, H, W, n_fg - int(0.02 * n_fg), cells)
        means = _sphere(g, cells, d)
        kappas = 20.0 + 180.0 * torch.rand(cells, generator=g, device=DEV, dtype=torch.float64)
        embs, masks = [], []
        for _ in range(case["frames"]):
            e, m = _frame(g, H, W, d, case["fill"], cells, 20.0, 200.0, 0.02, means, kappas, owner)
            embs.append(e)
            masks.append(m)
            t = torch.randn(cells, d, generator=g, device=DEV, dtype=torch.float64)
            t -= (t * means).sum(1, keepdim=True) * means
            means = math.cos(0.02) * means + math.sin(0.02) * t / t.norm(dim=1, keepdim=True)
        s.update(embs=embs, masks=masks, cfg=ms.ms_config_default(dim=d, **_options(case)))
    elif kind == "train":
        P, X0, target = _points(g, case["N"], case["M"], 16)
        s.update(P=P, X0=X0, target=target)
    else:
        P, X0, _ = _points(g, case["N"], case["M"], case["d"])
        s.update(P=P, X0=X0)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "blobs":
        r = ms.cluster(s["emb"], s["mask"], **_options(case))
        return {"labels": r.labels, "modes": r.modes, "support": r.stats["support"]}
    if kind == "frame":
        ctx = ms.ms_create(s["cfg"], s["emb"], s["mask"])
        k = ms.ms_run(ctx, s["labels"], s["modes"])
        ms.ms_destroy(ctx)
        return {"labels": s["labels"], "modes": s["modes"], "k": k}
    if kind == "host":
        k, _ = ms.ms_run_host(s["cfg"], s["emb"], s["mask"], s["labels"], s["modes"])
        return {"labels": s["labels"], "modes": s["modes"], "k": k}
    if kind == "batch":
        b = s["batch"]
        ms.ms_batch_run(b)
        for f, out in enumerate(s["modes"]):
            m = ms.ms_batch_modes(b, f)
            out[:m.shape[0]] = m
        return {"labels": list(b.labels), "modes": s["modes"]}
    if kind == "video":
        with ms.ms_video_create(s["cfg"], max(e.shape[0] for e in s["embs"])) as v:
            labels, n_start, n_modes = ms.ms_video_run(v, s["embs"], s["masks"])
        return {"labels": labels, "n_start": n_start, "n_modes": n_modes}
    if kind == "train":
        P = s["P"].detach().requires_grad_(True)
        X0 = s["X0"].detach().requires_grad_(True)
        x = vmf_mean_shift(P, X0, case["kappa"], case["T"], _precision(case))
        loss = ((x - s["target"]) ** 2).sum()
        loss.backward()
        return {"x": x.detach(), "loss": loss.detach(), "dP": P.grad, "dX0": X0.grad}
    x, counts = ms.ms_kernel_shift(s["P"], s["X0"], _DISTANCE[case["distance"]], _PROFILE[case["profile"]], case["h"],
                                   case["T"])
    return {"x": x, "counts": counts}


_DISTANCE = {"cosine": ms.MS_DIST_COSINE, "euclid": ms.MS_DIST_EUCLID}
_PROFILE = {"flat": ms.MS_PROFILE_FLAT, "epanechnikov": ms.MS_PROFILE_EPANECHNIKOV, "gaussian": ms.MS_PROFILE_GAUSSIAN}


def work(case):
    """Inputs read once, labels (or seeds and gradients) written once. Flops: the dense method's similarity and window
    sum, 4 d per pixel and seed-iteration; smooth kernel 64 per pair and step forward, 288 with the backward."""
    kind = case["kind"]
    if kind == "train":
        pairs = float(case["N"]) * case["M"] * case["T"]
        return {"bytes": 4.0 * 16 * (2 * case["N"] + 4 * case["M"]), "flops": (64 + 288) * pairs}
    if kind == "kshift":
        return {"bytes": 4.0 * case["d"] * (case["N"] + 2 * case["M"]), "flops": 4.0 * case["d"] * case["N"] * case["M"] * case["T"]}
    d = case["d"]
    if kind == "blobs":  # one round of n_initial seeds, a few iterations each
        return {"bytes": case["n"] * (4.0 * d + 4), "flops": 4.0 * d * case["n"] * case["n_initial"] * 3}
    if kind == "batch":
        fg = [float(n) for n in _batch_sizes(case)]
        px = [float(max(16, int(math.ceil(math.sqrt(2 * n)))) ** 2) for n in fg]
    else:
        px = [float(case["H"] * case["W"])] * case.get("frames", 1)
        fg = [case["fill"] * p for p in px]
    return {"bytes": sum(px) * 5 + sum(fg) * 4.0 * d, "flops": sum(4.0 * d * SEED_ITERS_PER_PIXEL * n * n for n in fg)}


# ---------------------------------------------------------------- 64 bits
def _seed_order(n, frame_id=0):
    """The fixed affine seed order (b + a j) mod n: a coprime to n nearest 0.618 n, b from SplitMix64."""
    if n <= 1:
        return np.zeros(n, dtype=np.int64)
    centre, a = int(math.floor(0.6180339887 * n + 0.5)), 1
    for off in range(n + 1):
        near = [v for v in (centre - off, centre + off) if 1 <= v < n and math.gcd(v, n) == 1]
        if near:
            a = near[0]
            break
    m = (1 << 64) - 1
    z = (frame_id + 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    z ^= z >> 31
    return ((z % n) + a * np.arange(n, dtype=np.int64)) % n


def _shift64(P, X, c, rows=1024):
    """Window sums and sizes of X over P (float64)."""
    Y, cnt = torch.empty_like(X), torch.empty(X.shape[0], dtype=torch.int64, device=X.device)
    for i in range(0, X.shape[0], rows):
        W = (X[i:i + rows] @ P.T) >= c
        cnt[i:i + rows] = W.sum(1)
        Y[i:i + rows] = W.double() @ P
    return Y, cnt


def _unit(v):
    return v / v.norm(dim=1, keepdim=True)


def _keep64(X, modes, c):
    """Which candidates (in rank order) the greedy merge keeps against the earlier modes and one another."""
    n = X.shape[0]
    kept = torch.zeros(n, dtype=torch.bool, device=X.device)
    gone = torch.zeros(n, dtype=torch.bool, device=X.device)
    Xn = _unit(X)
    for i in range(0, n, 4096):
        if modes.shape[0]:
            gone[i:i + 4096] = ((Xn[i:i + 4096] @ _unit(modes).T) >= c).any(1)
    for i in range(0, n, 4096):  # blocks in rank order; inside a block, sweeps
        blk = Xn[i:i + 4096]
        done = Xn[:i][kept[:i]]
        g = gone[i:i + 4096].clone()
        if done.shape[0]:
            g |= ((blk @ done.T) >= c).any(1)
        conflict = torch.tril((blk @ blk.T) >= c, -1)
        k = torch.zeros_like(g)
        while True:
            open_ = ~g & ~k
            if not bool(open_.any()):
                break
            k |= open_ & ~(conflict & open_[None, :]).any(1)
            g |= ~k & (conflict & k[None, :]).any(1)
        kept[i:i + 4096], gone[i:i + 4096] = k, g
    return kept


def _cluster64(emb, mask, c, n_initial, tol=1e-6, gamma=0.9, prob=0.99, low=2.0, high=8.0, max_iter=300):
    """Modes of the whole method in float64."""
    P = _unit((emb if mask is None else emb[mask.bool()]).double())
    n, d = P.shape
    order = torch.from_numpy(_seed_order(n)).to(P.device)
    covered = torch.zeros(n, dtype=torch.bool, device=P.device)
    modes = torch.zeros(0, d, dtype=torch.float64, device=P.device)
    support = torch.zeros(0, dtype=torch.int64, device=P.device)
    cursor, N = 0, n_initial
    while not bool(covered.all()):
        want = min(N, int((~covered).sum()))
        free = torch.nonzero(~covered[order[cursor:]]).reshape(-1)[:want]
        seeds = order[cursor + free]
        cursor += int(free[-1]) + 1
        covered[seeds] = True
        X = P[seeds].clone()
        active = torch.arange(want, device=P.device)
        conv = torch.zeros(want, dtype=torch.bool, device=P.device)
        size = torch.zeros(want, dtype=torch.int64, device=P.device)
        for _ in range(max_iter):
            Y, cnt = _shift64(P, X[active], c)
            ok = cnt > 0
            a, Y, size[active] = active[ok], _unit(Y[ok]), cnt
            stop = (Y - X[a]).norm(dim=1) < tol
            X[a] = Y
            conv[a[stop]] = True
            active = a[~stop]
            if int(conv.sum()) > gamma * want or active.numel() == 0:
                break
        cand = torch.nonzero(conv).reshape(-1)
        cand = cand[torch.argsort(size[cand], descending=True, stable=True)]
        cand = cand[_keep64(X[cand], modes, c)]
        new = X[cand]
        modes, support = torch.cat([modes, new]), torch.cat([support, size[cand]])
        for i in range(0, n, 16384):
            if new.shape[0]:
                covered[i:i + 16384] |= ((P[i:i + 16384] @ new.T) >= c).any(1)
        left, I = int((~covered).sum()), modes.shape[0]
        if I > 1:
            n_min = math.log(1.0 - math.exp(math.log(prob) / I)) / math.log(1.0 - 1.0 / I)
            N = 2 * N if N < low * n_min else N - math.ceil(n_min) if N > high * n_min else N
        N = max(1, min(N, max(1, left)))
    return modes


def _vmf64(P, X0, target, kappa, T):
    """x_T, the loss and both gradients by autograd in float64, a block of seeds at a time."""
    P = P.double().requires_grad_(True)
    X0 = X0.double().requires_grad_(True)
    xs, loss = [], 0.0
    rows = max(1, (1 << 23) // P.shape[0])
    for i in range(0, X0.shape[0], rows):
        x = X0[i:i + rows]
        for _ in range(T):
            x = _unit(torch.exp(kappa * (x @ P.T - 1.0)) @ P)
        part = ((x - target[i:i + rows].double()) ** 2).sum()
        part.backward()
        loss += part.detach()
        xs.append(x.detach())
    return {"x": torch.cat(xs), "loss": loss, "dP": P.grad, "dX0": X0.grad}


def _kshift64(P, X, distance, profile, h, T):
    P, X = P.double(), X.double()
    if distance == "cosine":
        P, X = _unit(P), _unit(X)
    for _ in range(T):
        for i in range(0, X.shape[0], 128):
            x = X[i:i + 128]
            dot = x @ P.T
            d2 = (1.0 - dot) ** 2 if distance == "cosine" else (x * x).sum(1)[:, None] + (P * P).sum(1) - 2.0 * dot
            t = d2 / (h * h)
            w = (t <= 1.0).double() if profile == "flat" else (1.0 - t).clamp(min=0.0) if profile == "epanechnikov" else torch.exp(-0.5 * t)
            y, sw = w @ P, w.sum(1, keepdim=True)
            y = _unit(y) if distance == "cosine" else y / sw
            X[i:i + 128] = torch.where(sw > 0, y, x)
    return {"x": X, "counts": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "video"):  # dozens of whole frames: minutes
        return None
    s = prepare(case, seed)
    if kind == "train":
        return _vmf64(s["P"], s["X0"], s["target"], case["kappa"], case["T"])
    if kind == "kshift":
        return _kshift64(s["P"], s["X0"], case["distance"], case["profile"], case["h"], case["T"])
    if case["d"] > 16 and kind != "blobs" and case["fill"] * case["H"] * case["W"] > 40000:
        return None  # tens of thousands of modes: over 20 s
    mask = s["mask"]
    modes = _cluster64(s["emb"].to(DEV), None if mask is None else mask.to(DEV), case["bandwidth"], case["n_initial"])
    if kind == "blobs":
        return {"labels": None, "modes": modes, "support": None}
    out = torch.zeros(s["modes"].shape, dtype=torch.float64, device=DEV)
    out[:modes.shape[0]] = modes
    return {"labels": None, "modes": out, "k": None}
