"""Workloads of the Haar-tSVD library, each one pass through its public entry points.

listed() and draw() name the cases, prepare() makes what a program holds before the call (device images,
parameters, networks), run() makes the call and returns everything it computes, work() counts what the call
cannot do without and exact() evaluates the same call in 64 bits with plain torch, from the paper's equations.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2512_23569_gb300 import hts

PS = 8
STEP = 4
FALLBACK = 2.0   # denoise_learned: accepted ratio of the learned and the estimated noise level
WINDOW = 128     # readout window of the learned map
LR = 2e-3


# ------------------------------------------------------------------ cases

def listed():
    return [
        # one small gray image at a time, known noise level: an interactive or streaming caller, where the
        # launches and the host path count
        dict(name="gray_small", kind="denoise", H=128, W=96, C=1, K=16, win=21, precision=0, sigma=25.0),
        # the certified plain form on the standard colour test size, noise level estimated
        dict(name="colour512_plain", kind="denoise", H=512, W=512, C=3, K=16, win=31, precision=0, sigma=-50.0),
        # exact groups with the tensor-core filter on an odd-sized photo crop, noise level estimated
        dict(name="colour_odd_exact_groups", kind="denoise", H=1021, W=771, C=3, K=16, win=31, precision=2,
             sigma=-30.0),
        # a UHD frame through the learned noise map and the precision form: the framework's default workload
        dict(name="learned_uhd", kind="learned", H=2160, W=3840, C=3, K=16, win=31, precision=1),
        # several images of mixed sizes, gray and colour, in one graph launch
        dict(name="batch_mixed", kind="batch", small=4, medium=4, large=2, huge=1, precision=1),
        # grouping alone, certified, with the paper's K = 32 on a gray image
        dict(name="match_gray_k32", kind="match", H=768, W=1024, C=1, K=32, win=21, precision=0),
        # grouping alone on the tensor cores, the largest image of the mixed sets
        dict(name="match_colour_tc", kind="match", H=1536, W=2048, C=3, K=16, win=31, precision=1),
        # noise level and basis of a 1024 x 1024 colour image, for a caller that decides what to do with it
        dict(name="sigma_colour1024", kind="sigma", H=1024, W=1024, C=3, K=16, win=31, precision=1, sigma=20.0),
        # the network's noise map alone
        dict(name="cnn_map", kind="cnn_map", H=1536, W=2048, C=3),
        # one training step of the noise map: eight 256 x 256 colour crops, as its training runs it
        dict(name="cnn_train", kind="cnn_train", H=256, W=256, C=3, batch=8),
        # one training step of the enhancement network on 4096 pairs of mean patches
        dict(name="fcn_train", kind="fcn_train", n=4096, C=3, K=16),
        # denoising with the enhancement network
        dict(name="ra_colour512", kind="ra", H=512, W=512, C=3, K=16, win=31, precision=2, sigma=50.0),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, pixels):
    """H, W of an image of at most `pixels` pixels, sides from `lo`, aspect within 2:1, any parity."""
    n = math.exp(rng.uniform(math.log(lo * lo), math.log(pixels)))
    a = math.exp(rng.uniform(-0.5, 0.5) * math.log(2.0))
    return max(lo, int(math.sqrt(n * a))), max(lo, int(math.sqrt(n / a)))


def draw(rng):
    kind = rng.choice(["denoise", "denoise", "denoise", "learned", "batch", "match", "match", "sigma", "cnn_map",
                       "cnn_train", "fcn_train", "ra"])
    C = rng.choice([1, 3])
    win = 31 if C == 3 else 21
    K = rng.choice([8, 16, 16, 32])
    if kind == "denoise":
        precision = rng.choice([0, 1, 2])
        H, W = _size(rng, 64, 8.0e6 if precision == 1 else 1.6e6)
        sigma = round(rng.uniform(10.0, 75.0), 1) * rng.choice([1, -1])
        return dict(kind=kind, H=H, W=W, C=C, K=K, win=win, precision=precision, sigma=sigma)
    if kind == "learned":
        H, W = _size(rng, 192, 8.0e6)
        return dict(kind=kind, H=H, W=W, C=C, K=16, win=win, precision=1)
    if kind == "batch":
        return dict(kind=kind, small=rng.randint(1, 6), medium=rng.randint(0, 6), large=rng.randint(0, 3), huge=0,
                    precision=rng.choice([1, 1, 2]))
    if kind == "match":
        precision = rng.choice([0, 1])
        H, W = _size(rng, 64, 8.0e6 if precision else 1.6e6)
        return dict(kind=kind, H=H, W=W, C=C, K=K, win=win, precision=precision)
    if kind == "sigma":
        H, W = _size(rng, 96, 4.0e6)
        return dict(kind=kind, H=H, W=W, C=C, K=16, win=win, precision=1, sigma=round(rng.uniform(10.0, 75.0), 1))
    if kind == "cnn_map":
        H, W = _size(rng, 64, 8.0e6)
        return dict(kind=kind, H=H, W=W, C=C)
    if kind == "cnn_train":
        H, W = _size(rng, 48, 1.3e5)
        return dict(kind=kind, H=H, W=W, C=C, batch=rng.randint(1, 8))
    if kind == "fcn_train":
        return dict(kind=kind, n=_spread(rng, 100, 16384), C=C, K=K)
    H, W = _size(rng, 64, 4.0e5)
    return dict(kind=kind, H=H, W=W, C=C, K=16, win=win, precision=rng.choice([1, 2]),
                sigma=round(rng.uniform(30.0, 75.0), 1))


# ----------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed & 0x7FFFFFFF)


def _clean(H, W, C, g):
    """Flat ground with rectangles, disks and two gratings, on [0, 255]; channels share the geometry."""
    r = torch.rand(256, generator=g, device="cuda").cpu().tolist()
    at = iter(r)
    u = lambda lo, hi: lo + (hi - lo) * next(at)  # noqa: E731
    img = torch.full((H, W), u(0, 255), device="cuda")
    yy = torch.arange(H, device="cuda", dtype=torch.float32)[:, None]
    xx = torch.arange(W, device="cuda", dtype=torch.float32)[None, :]
    for _ in range(20):
        y0, x0 = int(u(0, H)), int(u(0, W))
        img[y0:y0 + 2 + int(u(0, H / 3)), x0:x0 + 2 + int(u(0, W / 3))] = u(0, 255)
    for _ in range(10):
        cy, cx, rad, v = u(0, H), u(0, W), u(4, max(5.0, min(H, W) / 6)), u(0, 255)
        img = torch.where((yy - cy) ** 2 + (xx - cx) ** 2 <= rad * rad, v, img)
    for _ in range(2):
        period, ang, amp = u(6, 20), u(0, math.pi), u(20, 60)
        img = img + amp * torch.sin((2 * math.pi / period) * (math.cos(ang) * xx + math.sin(ang) * yy))
    img = img.clamp(0, 255)
    gains = [1.0] if C == 1 else [u(0.8, 1.2) for _ in range(3)]
    return torch.stack([(img * s).clamp(0, 255) for s in gains])


def _noisy(H, W, C, sigma, seed):
    g = _gen(seed)
    x = _clean(H, W, C, g)
    return (x + sigma * torch.randn(x.shape, generator=g, device="cuda")).contiguous()


def _noisy_varying(H, W, C, seed):
    """Signal-dependent noise plus read noise that ramps across the image from 2 to 28."""
    g = _gen(seed)
    x = _clean(H, W, C, g)
    ramp = torch.linspace(2.0, 28.0, W, device="cuda")[None, None, :]
    y = 0.01 * torch.poisson(x / 0.01, generator=g) + ramp * torch.randn(x.shape, generator=g, device="cuda")
    return y.contiguous()


def _cnn_theta(C, seed):
    """Weights of the noise-map network about a level of 15 on the [0, 255] scale."""
    rng = np.random.default_rng(seed)
    parts = []
    widths = [C, 32, 32, 32, 32, 1]
    for l in range(5):
        ci, co = widths[l], widths[l + 1]
        s = math.sqrt(2.0 / (9 * ci)) if l < 4 else 0.03
        parts.append(s * rng.standard_normal(co * ci * 9))
        parts.append(np.full(co, math.log(15.0)) if l == 4 else 0.02 * rng.standard_normal(co))
    return np.concatenate(parts).astype(np.float32)


def _fcn_dims(C):
    return [(C * 64 + 16) // 16 * 16, 128, 128, C * 64]


def _fcn_theta(C, seed):
    rng = np.random.default_rng(seed)
    d = _fcn_dims(C)
    parts = []
    for l in range(3):
        s = math.sqrt(2.0 / d[l]) * (0.1 if l == 2 else 1.0)
        parts.append(s * rng.standard_normal(d[l] * d[l + 1]))
        parts.append(0.01 * rng.standard_normal(d[l + 1]))
    return np.concatenate(parts).astype(np.float32)


def _batch_specs(case):
    """(H, W, C, sigma) of a batch: the mixed sizes, alternately gray and colour."""
    sizes = ([(256, 256)] * case["small"] + [(384, 512)] * case["medium"] + [(768, 1024)] * case["large"] +
             [(1536, 2048)] * case["huge"])
    return [(h, w, 3 if i % 2 == 0 else 1, 10.0 + (37 * i) % 65) for i, (h, w) in enumerate(sizes)]


def _pairs(case, seed):
    """Noisy and clean mean-patch coordinates: sparse coefficients, and the noise of a mean of K patches."""
    n, C = case["n"], case["C"]
    g = _gen(seed)
    sigma = 30.0 + 45.0 * torch.rand(n, generator=g, device="cuda")
    clean = torch.randn((n, C * 64), generator=g, device="cuda") * 40.0
    clean = clean * (torch.rand((n, C * 64), generator=g, device="cuda") < 0.15)
    clean[:, 0] = 400.0 + 400.0 * torch.rand(n, generator=g, device="cuda")
    noise = torch.randn((n, C * 64), generator=g, device="cuda")
    noisy = clean + noise * (sigma / math.sqrt(case["K"]))[:, None]
    return noisy.contiguous(), clean.contiguous(), sigma.contiguous()


def _crops(case, seed):
    H, W, C = case["H"], case["W"], case["C"]
    xs = [_noisy_varying(H, W, C, seed * 16 + i) for i in range(case["batch"])]
    n = _nref(H, W)
    ts = [math.log(15.0) + 0.5 * torch.randn(n, generator=_gen(seed * 16 + i + 7), device="cuda")
          for i in range(case["batch"])]
    return xs, ts


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if "win" in case:
        s["p"] = hts.params(K=case["K"], win=case["win"], precision=case["precision"])
    if kind in ("denoise", "sigma", "ra"):
        s["x"] = _noisy(case["H"], case["W"], case["C"], abs(case["sigma"]), seed)
    elif kind in ("learned", "cnn_map"):
        s["x"] = _noisy_varying(case["H"], case["W"], case["C"], seed)
    elif kind == "match":
        s["x"] = _noisy(case["H"], case["W"], case["C"], 25.0, seed)
    if kind in ("learned", "cnn_map", "cnn_train"):
        s["net"] = hts.Cnn(case["C"])
        s["net"].set_params(_cnn_theta(case["C"], seed))
        s["net"].window = WINDOW
    if kind == "cnn_train":
        s["p"] = hts.params()
        s["xs"], s["ts"] = _crops(case, seed)
    if kind in ("fcn_train", "ra"):
        s["fcn"] = hts.Fcn(case["C"], case["K"])
        s["fcn"].set_params(_fcn_theta(case["C"], seed))
    if kind == "fcn_train":
        s["pairs"] = _pairs(case, seed)
    if kind == "batch":
        specs = _batch_specs(case)
        s["xs"] = [_noisy(h, w, c, sg, seed * 64 + i) for i, (h, w, c, sg) in enumerate(specs)]
        s["sigmas"] = [sg for _, _, _, sg in specs]
        s["p"] = hts.params(K=16, win=31, precision=case["precision"])
        s["per"] = [hts.params(K=16, win=31 if c == 3 else 21, precision=case["precision"]) for _, _, c, _ in specs]
    return s


# -------------------------------------------------------------------- run

def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "denoise":
        return hts.denoise(s["x"], sigma=case["sigma"] if case["sigma"] > 0 else None, p=s["p"])
    if kind == "learned":
        return hts.denoise_learned(s["x"], s["net"], p=s["p"], fallback_factor=FALLBACK)
    if kind == "ra":
        return hts.denoise_ra(s["x"], s["fcn"], sigma=case["sigma"], p=s["p"])
    if kind == "batch":
        return hts.denoise_batch(s["xs"], s["sigmas"], p=s["p"], per_image=s["per"])
    if kind == "match":
        return list(hts.match(s["x"], p=s["p"]))
    if kind == "sigma":
        basis = hts.estimate_basis(s["x"], p=s["p"])
        sigma, info = hts.estimate_sigma(s["x"], p=s["p"], basis=basis)
        return {"eigvals": basis.read()[1], "sigma": sigma, "votes": info["votes"], "adjusted": info["adjusted"]}
    if kind == "cnn_map":
        return s["net"].log_sigma_map(s["x"])
    if kind == "cnn_train":
        net = s["net"]
        net.zero_grad()
        for x, t in zip(s["xs"], s["ts"]):
            net.accumulate_grad(x, t, p=s["p"])
        net.adam_step(LR)
        return {"grad": net.get_grad(), "loss": net.take_loss(), "params": net.get_params()}
    fcn = s["fcn"]
    fcn.zero_grad()
    fcn.accumulate_grad(*s["pairs"])
    fcn.adam_step(LR)
    return {"grad": fcn.get_grad(), "loss": fcn.take_loss(), "params": fcn.get_params()}


# ------------------------------------------------------------------- work

def _nref(H, W):
    return len(_grid(H)) * len(_grid(W))


def _work_match(H, W, C, win):
    return 3.0 * 64 * _nref(H, W) * win * win


def _work_filter(H, W, C, K):
    per = 2.0 * (K * (10240 if C == 3 else 2048) + C * 64 * 4 * (K - 1))
    return per * _nref(H, W)


def _work_basis(H, W, C):
    return 2.0 * _nref(H, W) * 2 * 8 * (36 if C == 1 else 300)


def _work_cnn(H, W, C):
    return 2.0 * 9 * H * W * (C * 32 + 3 * 32 * 32 + 32)


def _work_vote(H, W, C, K):
    return 5.0 * C * 64 * K * math.log2(K) * _nref(H, W)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for h, w, c, _ in _batch_specs(case):
            total["bytes"] += 8.0 * c * h * w
            total["flops"] += (_work_match(h, w, c, 31 if c == 3 else 21) + _work_filter(h, w, c, 16) +
                               _work_basis(h, w, c))
        return total
    C = case["C"]
    if kind == "fcn_train":
        d = _fcn_dims(C)
        p = sum(d[i] * d[i + 1] for i in range(3))
        flops = 2.0 * case["n"] * (3 * p - d[0] * d[1])
        return {"bytes": case["n"] * (8.0 * C * 64 + 4) + 20.0 * (p + sum(d[1:])), "flops": flops}
    H, W = case["H"], case["W"]
    image = 4.0 * C * H * W
    if kind == "cnn_train":
        n = case["batch"]
        return {"bytes": n * (image + 4.0 * _nref(H, W)) + 20.0 * hts.load().hts_cnn_num_params(C),
                "flops": n * (3 * _work_cnn(H, W, C) - 2.0 * 9 * H * W * C * 32)}
    if kind == "cnn_map":
        return {"bytes": image + 4.0 * H * W, "flops": _work_cnn(H, W, C)}
    if kind == "match":
        return {"bytes": image + _nref(H, W) * (4.0 * case["K"] + 1), "flops": _work_match(H, W, C, case["win"])}
    flops = _work_match(H, W, C, case["win"]) + _work_basis(H, W, C)
    if kind == "sigma":
        return {"bytes": image, "flops": flops + _work_vote(H, W, C, case["K"])}
    flops += _work_filter(H, W, C, case["K"])
    if kind == "learned":
        flops += _work_cnn(H, W, C) + _work_vote(H, W, C, case["K"])
    elif case["sigma"] < 0:
        flops += _work_vote(H, W, C, case["K"])
    if kind == "ra":
        d = _fcn_dims(C)
        flops += 2.0 * _nref(H, W) * sum(d[i] * d[i + 1] for i in range(3))
    return {"bytes": 2 * image, "flops": flops}


# ------------------------------------------- the same in 64 bits, plain torch

def _grid(n):
    g = list(range(0, n - PS + 1, STEP))
    return g if g[-1] == n - PS else g + [n - PS]


def _grids(H, W):
    return torch.tensor(_grid(H), device="cuda"), torch.tensor(_grid(W), device="cuda")


def _patch_sums(a, ys, xs):
    """Sums of the 8 x 8 patches of `a` whose corners are ys x xs."""
    cols = sum(a[:, xs + v] for v in range(PS))
    return sum(cols[ys + u, :] for u in range(PS))


def _groups(img, K, win):
    """Raster indices of every group: the patch, then its K - 1 nearest in the window (Eq. 9)."""
    C, H, W = img.shape
    ys, xs = _grids(H, W)
    R = win // 2
    n = len(ys) * len(xs)
    planes = [img[0]] if C == 1 else [img[1], (img[0] + img[1]) + img[2]]
    green = None
    if C == 3:
        nr, ng, nb = (_patch_sums(img[c] ** 2, ys, xs).sqrt() for c in range(3))
        green = ng >= torch.maximum(nr / 1.2, nb / 1.2)
    dist = torch.full((n, win * win), math.inf, dtype=torch.float64, device="cuda")
    for o in range(win * win):
        dy, dx = o // win - R, o % win - R
        if dy == 0 and dx == 0:
            continue
        yok = (ys + dy >= 0) & (ys + dy <= H - PS)
        xok = (xs + dx >= 0) & (xs + dx <= W - PS)
        ya, xa = ys[yok], xs[xok]
        y0, x0 = max(0, -dy), max(0, -dx)
        y1, x1 = min(H, H - dy), min(W, W - dx)
        d = [_patch_sums((p[y0:y1, x0:x1] - p[y0 + dy:y1 + dy, x0 + dx:x1 + dx]) ** 2, ya - y0, xa - x0)
             for p in planes]
        ok = yok[:, None] & xok[None, :]
        dist[ok.reshape(-1), o] = (d[0] if C == 1 else torch.where(green[ok].view(len(ya), len(xa)), d[0],
                                                                   d[1])).reshape(-1)
    ref = (ys[:, None] * W + xs[None, :]).reshape(-1)
    idx = torch.empty((n, K), dtype=torch.int64, device="cuda")
    idx[:, 0] = ref
    for a in range(0, n, 65536):
        o = torch.topk(dist[a:a + 65536], K - 1, largest=False, sorted=True).indices
        idx[a:a + 65536, 1:] = ref[a:a + 65536, None] + (o // win - R) * W + (o % win - R)
    return idx


def _slices(img):
    """Channel DFT (unitary): the real slice, and for colour the complex one (its conjugate is implied)."""
    if img.shape[0] == 1:
        return [img[0].to(torch.complex128)]
    w = torch.exp(torch.tensor(-2j * math.pi / 3, dtype=torch.complex128, device="cuda"))
    s = 1.0 / math.sqrt(3.0)
    z = img.to(torch.complex128)
    return [s * (z[0] + z[1] + z[2]), s * (z[0] + w * z[1] + w * w * z[2])]


def _basis(img):
    """Eigenvectors and eigenvalues of the row and column covariances of all patches (Eq. 11)."""
    C, H, W = img.shape
    ys, xs = _grids(H, W)
    uv, ev = [], []
    for z in _slices(img):
        row = torch.zeros((PS, PS), dtype=torch.complex128, device="cuda")
        col = torch.zeros((PS, PS), dtype=torch.complex128, device="cuda")
        lines = torch.stack([z[:, xs + v] for v in range(PS)])  # [v][H][nx]
        for a in range(PS):
            for b in range(a, PS):
                row[a, b] = sum((lines[v][ys + a] * lines[v][ys + b].conj()).sum() for v in range(PS))
                row[b, a] = row[a, b].conj()
                col[a, b] = sum((lines[a][ys + u].conj() * lines[b][ys + u]).sum() for u in range(PS))
                col[b, a] = col[a, b].conj()
        pair, vals = [], []
        for m in (row, col):
            lam, q = torch.linalg.eigh(m.real if len(uv) == 0 else m)
            q = q.to(torch.complex128)
            top = q.abs().argmax(dim=0)  # phases: each eigenvector's largest entry real and positive
            lead = q[top, torch.arange(PS, device="cuda")]
            pair.append(q * (lead.conj() / lead.abs())[None, :])
            vals.append(lam)
        uv.append(pair)
        ev.append(torch.stack(vals))
    return uv, torch.stack(ev)


def _transform(uv, C):
    """The orthonormal map of a patch to its coefficients [S1 | sqrt2 Re S2 | sqrt2 Im S2] (Eq. 4-5, 19)."""
    kron = [torch.kron(u.conj().T.contiguous(), v.T.contiguous()) for u, v in uv]
    if C == 1:
        return kron[0].real.contiguous()
    w = np.exp(-2j * math.pi / 3)
    s = 1.0 / math.sqrt(3.0)
    f0 = torch.cat([s * kron[0].real] * 3, dim=1)
    f1 = torch.cat([s * complex(w ** t) * kron[1] for t in range(3)], dim=1)
    return torch.cat([f0, math.sqrt(2.0) * f1.real, math.sqrt(2.0) * f1.imag], dim=0).contiguous()


def _haar(K):
    h = torch.ones((1, 1), dtype=torch.float64)
    while h.shape[0] < K:
        h = torch.cat([torch.kron(h, torch.tensor([[1.0, 1.0]], dtype=torch.float64)),
                       torch.kron(torch.eye(h.shape[0], dtype=torch.float64),
                                  torch.tensor([[1.0, -1.0]], dtype=torch.float64))]) / math.sqrt(2.0)
    return h.cuda()


def _offsets(H, W, C):
    o = torch.arange(PS, device="cuda")
    return (torch.arange(C, device="cuda")[:, None, None] * H * W + o[None, :, None] * W + o[None, None, :]).reshape(-1)


def _votes(img, idx):
    """Groups whose rank position of the alternating eigenvalue is small (Eq. 22-23)."""
    C, H, W = img.shape
    K = idx.shape[1]
    off, flat = _offsets(H, W, C), img.reshape(-1)
    votes = 0
    for a in range(0, len(idx), 8192):
        lam = torch.fft.fft(flat[idx[a:a + 8192, :, None] + off], dim=1).abs().square().sum(dim=2)
        rank = 1 + (lam < lam[:, K // 2:K // 2 + 1]).sum(dim=1)
        votes += int((rank <= 13.0 * K / 32.0).sum())
    return votes


def _sigma(img, ev, idx):
    n = len(idx)
    s2 = max(float(ev.min()), 0.0) / (PS * n) / (1.0 - 1.0 / math.sqrt(n)) ** 2
    votes = _votes(img, idx)
    adjusted = int(2 * votes > n)
    return math.sqrt(s2) / (1.2 if adjusted else 1.0), votes, adjusted


def _filter(img, idx, T, sigma, refine=None):
    """Transform, threshold, inverse and plain average (Eq. 19-21, Alg. 1 step 3); sigma: one or one per group."""
    C, H, W = img.shape
    K = idx.shape[1]
    off, flat, h = _offsets(H, W, C), img.reshape(-1), _haar(K)
    tau = torch.as_tensor(sigma, dtype=torch.float64, device="cuda").expand(len(idx)) * math.sqrt(
        2.0 * math.log(C * K * PS * PS))
    acc = torch.zeros(C * H * W, dtype=torch.float64, device="cuda")
    cnt = torch.zeros(C * H * W, dtype=torch.float64, device="cuda")
    for a in range(0, len(idx), 8192):
        at = idx[a:a + 8192, :, None] + off
        coef = torch.einsum("hk,nkd->nhd", h, flat[at] @ T.T)
        t = tau[a:a + 8192, None, None]
        mag = coef[:, :, :64].abs() >= t
        if C == 3:
            pair = torch.hypot(coef[:, :, 64:128], coef[:, :, 128:]) >= math.sqrt(2.0) * t
            mag = torch.cat([mag, pair, pair], dim=2)
        kept = coef * mag
        if refine is not None:
            kept[:, 0] = refine(coef[:, 0] / math.sqrt(K), K) * math.sqrt(K)
        est = torch.einsum("hk,nhd->nkd", h, kept) @ T
        acc.index_add_(0, at.reshape(-1), est.reshape(-1))
        cnt.index_add_(0, at.reshape(-1), torch.ones_like(est).reshape(-1))
    return (acc / cnt).view(C, H, W)


def _cnn_layers(theta, C):
    t = torch.as_tensor(theta, dtype=torch.float64, device="cuda")
    widths, out, o = [C, 32, 32, 32, 32, 1], [], 0
    for l in range(5):
        ci, co = widths[l], widths[l + 1]
        w = t[o:o + co * ci * 9].view(co, ci, 3, 3)
        o += co * ci * 9
        out.append((w, t[o:o + co]))
        o += co
    return out


def _cnn_forward(layers, img):
    x = img / 255.0
    for l, (w, b) in enumerate(layers):
        H, W = x.shape[1:]
        xp = torch.nn.functional.pad(x, (1, 1, 1, 1))
        z = b[:, None].expand(-1, H * W)
        for ky in range(3):
            for kx in range(3):
                z = z + w[:, :, ky, kx] @ xp[:, ky:ky + H, kx:kx + W].reshape(x.shape[0], -1)
        x = (torch.relu(z) if l < 4 else z).view(-1, H, W)
    return x[0]


def _window_sigma(m):
    """exp of the mean of the map over the readout window of every reference patch, cut to the image."""
    H, W = m.shape
    ys, xs = _grids(H, W)
    c = torch.zeros((H + 1, W + 1), dtype=torch.float64, device="cuda")
    c[1:, 1:] = m.cumsum(0).cumsum(1)
    y0, x0 = ys + 4 - WINDOW // 2, xs + 4 - WINDOW // 2
    y1, x1 = (y0 + WINDOW).clamp(max=H), (x0 + WINDOW).clamp(max=W)
    y0, x0 = y0.clamp(min=0), x0.clamp(min=0)
    s = c[y1][:, x1] - c[y0][:, x1] - c[y1][:, x0] + c[y0][:, x0]
    return torch.exp(s / ((y1 - y0)[:, None] * (x1 - x0)[None, :])).reshape(-1)


def _adam(theta, grad):
    return theta - LR * grad / (grad.abs() + 1e-8)


def _fcn_layers(theta, C):
    t = torch.as_tensor(theta, dtype=torch.float64, device="cuda")
    d, out, o = _fcn_dims(C), [], 0
    for l in range(3):
        w = t[o:o + d[l] * d[l + 1]].view(d[l + 1], d[l])
        o += d[l] * d[l + 1]
        out.append((w, t[o:o + d[l + 1]]))
        o += d[l + 1]
    return out


def _fcn_forward(layers, coefs, sigma, K):
    """The network's output in units of the mean patch's noise level, and that unit."""
    unit = (sigma / math.sqrt(K))[:, None]
    x = coefs / unit
    x = torch.cat([x / (1.0 + x.abs() / 16.0), sigma[:, None] / 255.0], dim=1)
    x = torch.nn.functional.pad(x, (0, layers[0][0].shape[1] - x.shape[1]))
    for l, (w, b) in enumerate(layers):
        x = x @ w.T + b
        x = torch.relu(x) if l < 2 else x
    return x, unit


def _exact_denoise(x, K, win, sigma, theta=None):
    img = x.double()
    idx = _groups(img, K, win)
    uv, ev = _basis(img)
    C = img.shape[0]
    level = sigma if sigma > 0 else _sigma(img, ev, idx)[0]
    refine = None
    if theta is not None:
        layers = _fcn_layers(theta, C)

        def refine(c, k):
            out, unit = _fcn_forward(layers, c, torch.full((len(c),), level, dtype=torch.float64, device="cuda"), k)
            return c + unit * out

    return _filter(img, idx, _transform(uv, C), level, refine)


def exact(case, seed):
    kind = case["kind"]
    if kind == "denoise":
        x = _noisy(case["H"], case["W"], case["C"], abs(case["sigma"]), seed)
        return _exact_denoise(x, case["K"], case["win"], case["sigma"])
    if kind == "ra":
        x = _noisy(case["H"], case["W"], case["C"], case["sigma"], seed)
        return _exact_denoise(x, case["K"], case["win"], case["sigma"], _fcn_theta(case["C"], seed))
    if kind == "batch":
        return [_exact_denoise(_noisy(h, w, c, sg, seed * 64 + i), 16, 31 if c == 3 else 21, sg)
                for i, (h, w, c, sg) in enumerate(_batch_specs(case))]
    if kind == "sigma":
        img = _noisy(case["H"], case["W"], case["C"], case["sigma"], seed).double()
        _, ev = _basis(img)
        sigma, votes, adjusted = _sigma(img, ev, _groups(img, case["K"], case["win"]))
        return {"eigvals": ev, "sigma": sigma, "votes": votes, "adjusted": adjusted}
    if kind in ("cnn_map", "learned"):
        img = _noisy_varying(case["H"], case["W"], case["C"], seed).double()
        m = _cnn_forward(_cnn_layers(_cnn_theta(case["C"], seed), case["C"]), img)
        if kind == "cnn_map":
            return m
        idx = _groups(img, case["K"], case["win"])
        uv, ev = _basis(img)
        level, estimate = _window_sigma(m), _sigma(img, ev, idx)[0]
        ratio = float(torch.exp(torch.log(level / estimate).mean()))
        if not 1.0 / FALLBACK <= ratio <= FALLBACK:
            level = estimate
        return _filter(img, idx, _transform(uv, case["C"]), level)
    if kind == "cnn_train":
        theta = torch.as_tensor(_cnn_theta(case["C"], seed), dtype=torch.float64, device="cuda").requires_grad_()
        ys, xs = _grids(case["H"], case["W"])
        loss = 0.0
        for x, t in zip(*_crops(case, seed)):
            m = _cnn_forward(_cnn_layers(theta, case["C"]), x.double())
            loss = loss + ((m[ys + 4][:, xs + 4].reshape(-1) - t.double()) ** 2).mean()
        loss.backward()
        return {"grad": theta.grad, "loss": float(loss), "params": _adam(theta.detach(), theta.grad)}
    if kind == "fcn_train":
        theta = torch.as_tensor(_fcn_theta(case["C"], seed), dtype=torch.float64, device="cuda").requires_grad_()
        noisy, clean, sigma = (t.double() for t in _pairs(case, seed))
        out, unit = _fcn_forward(_fcn_layers(theta, case["C"]), noisy, sigma, case["K"])
        loss = ((out - (clean - noisy) / unit) ** 2).mean()
        loss.backward()
        return {"grad": theta.grad, "loss": float(loss), "params": _adam(theta.detach(), theta.grad)}
    return None  # groups are whole numbers
