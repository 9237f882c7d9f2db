"""The work that users of this framework have it do, as cases to be measured.

A case is a dict of plain values.  Its "op" names the public call:

  search   mf.search: one matched-filter search of a residual stack;
  rescore  mf.rescore_topk: the candidate list of a search and its FP64
           re-score from the master stack;
  detect   mf.detect: local-sigma normalisation and detections of a score map;
  refit    mf.background_refit: the per-pixel background fit that makes the
           residual stack;
  batch    mf.Batch.run: uneven cutouts in one graph-captured launch.

Inputs follow the repository's synthetic sky: log-normal noise, clustered
masks of saturated stars, linear movers, scattered light with jitter terms.
"""
import math

import numpy as np
import torch

import paper_2209_09848_gb300 as mf
from paper_2209_09848_gb300 import synth

DEV = "cuda"
DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}
KINDS = {"gauss": 0, "shiftstack": 2}
SIGMA_PRF = 0.7


def _search(name, T, H, W, nx, ny, vmax, dtype="f32", prf="gauss", mask=0.01, frames=False, cube=False):
    return dict(name=name, op="search", T=T, H=H, W=W, nx=nx, ny=ny, vmax=vmax, dtype=dtype, prf=prf, mask=mask,
                frames=frames, cube=cube)


def listed():
    return [
        # the README's first search and the tests' small configuration: a
        # postage stamp, every score wanted; launches and latency count
        _search("search-stamp", 32, 128, 128, 4, 4, 0.15, mask=0.0, cube=True),
        # one ragged cutout around a sky position, with the real frame times
        # (a downlink gap) and pointing jitter
        _search("search-cutout-jitter", 333, 301, 277, 6, 9, 0.1, mask=0.02, frames=True),
        # the paper's search: one TESS CCD for one sector, 100 velocities
        _search("search-ccd", 1000, 2048, 2048, 10, 10, 0.1),
        # a fine velocity grid over a stack kept in bf16 to halve its memory
        _search("search-bf16-fine-grid", 600, 512, 512, 20, 20, 0.1, dtype="bf16"),
        # the shift-stack comparison of the paper: one tap per frame
        _search("search-shiftstack", 1000, 1024, 1024, 10, 10, 0.1, prf="shiftstack"),
        # a measured, non-separable PSF given as explicit footprints
        _search("search-measured-psf", 60, 500, 421, 6, 4, 0.3, prf="custom", mask=0.02),
        # the candidate list that follows a search
        dict(name="rescore-top4096", op="rescore", T=1000, H=1024, W=1024, nx=10, ny=10, vmax=0.1, k_top=4096,
             mask=0.01),
        # detections of a whole CCD's score map with the paper's 255 x 255 window
        dict(name="detect-ccd", op="detect", H=2048, W=2048, window=255, max_out=4096, zmap=True),
        # detections of one cutout's score map, odd sizes
        dict(name="detect-cutout", op="detect", H=301, W=277, window=63, max_out=256, zmap=False),
        # the background fit of a whole CCD and sector
        dict(name="refit-ccd", op="refit", T=1000, H=2048, W=2048, n=64, iterations=10, delta=1.345),
        # the same for one cutout over part of a sector
        dict(name="refit-cutout", op="refit", T=203, H=317, W=411, n=16, iterations=10, delta=1.345),
        # a batch of uneven cutouts, FP32, bf16 and scaled fp16 mixed
        dict(name="batch-cutouts", op="batch", items=12, side_lo=128, side_hi=384, t_lo=100, t_hi=500, k_lo=16,
             k_hi=100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["search"] * 5 + ["rescore", "detect", "detect", "refit", "refit", "batch"])
    if op == "search":
        prf = rng.choice(["gauss", "gauss", "gauss", "shiftstack", "custom"])
        H, W = _log(rng, 64, 1600), _log(rng, 64, 1600)
        T = _log(rng, 8, 160 if prf == "custom" else 1300)
        nx, ny = _log(rng, 1, 20), _log(rng, 1, 20)
        while H * W * T * nx * ny > (1e10 if prf == "custom" else 1e11):
            H, W = max(64, H * 3 // 4), max(64, W * 3 // 4)
            T, nx = max(8, T * 4 // 5), max(1, nx * 3 // 4)
        return dict(op="search", T=T, H=H, W=W, nx=nx, ny=ny, vmax=rng.choice([0.05, 0.1, 0.1, 0.3]),
                    dtype=rng.choice(["f32", "f32", "bf16", "fp16"]), prf=prf, mask=rng.choice([0.0, 0.01, 0.03]),
                    frames=prf != "custom" and rng.random() < 0.3, cube=nx * ny * H * W < 2e6)
    if op == "rescore":
        H, W = _log(rng, 100, 1200), _log(rng, 100, 1200)
        return dict(op="rescore", T=_log(rng, 30, 1200), H=H, W=W, nx=rng.randint(2, 10), ny=rng.randint(2, 10),
                    vmax=0.1, k_top=min(_log(rng, 16, 16384), H * W // 4), mask=0.01)
    if op == "detect":
        H, W = _log(rng, 60, 2048), _log(rng, 60, 2048)
        return dict(op="detect", H=H, W=W, window=rng.choice([31, 63, 127, 255, 255]), max_out=_log(rng, 64, 16384),
                    zmap=rng.random() < 0.5)
    if op == "refit":
        return dict(op="refit", T=_log(rng, 30, 1300), H=_log(rng, 64, 1024), W=_log(rng, 64, 1024),
                    n=rng.choice([8, 16, 64]), iterations=rng.randint(4, 12), delta=rng.choice([1.0, 1.345, 2.0]))
    return dict(op="batch", items=rng.randint(3, 16), side_lo=64, side_hi=_log(rng, 100, 400), t_lo=30,
                t_hi=_log(rng, 60, 500), k_lo=4, k_hi=_log(rng, 9, 120))


# ---------------------------------------------------------------- inputs ---

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _mask(H, W, frac, g):
    """Clustered 3 x 3 .. 7 x 7 blobs over about `frac` of the pixels."""
    if not frac:
        return None
    m = torch.zeros((1, 1, H, W), device=DEV)
    for r in (1, 2, 3):
        c = (torch.rand((1, 1, H, W), generator=g, device=DEV) < frac / 3 / (2 * r + 1) ** 2).float()
        m = torch.maximum(m, torch.nn.functional.max_pool2d(c, 2 * r + 1, 1, r))
    return m[0, 0].to(torch.uint8).contiguous()


def _sky(T, H, W, mask, dtype, seed):
    """Residual stack, noise map, mask and frame scales (fp16 only)."""
    g = _gen(seed)
    sigma = torch.exp(0.3 * torch.randn((H, W), generator=g, device=DEV))
    m = _mask(H, W, mask, g)
    res = torch.empty((T, H, W), device=DEV)
    for t0 in range(0, T, 64):
        res[t0:t0 + 64].normal_(generator=g).mul_(sigma)
    rng = np.random.default_rng(seed)
    n = max(1, min(200, H * W // 16384))
    ang, speed = rng.uniform(0, 2 * np.pi, n), rng.uniform(0.003, 0.1, n)
    movers = np.stack([rng.uniform(0, H, n), rng.uniform(0, W, n), speed * np.sin(ang), speed * np.cos(ang),
                       rng.uniform(0.05, 1.0, n)], 1)
    for i in range(n):  # one at a time: where two meet, the order of the sums is theirs
        synth.add_movers_torch(res, movers[i:i + 1], SIGMA_PRF)
    scale = None
    if dtype == "fp16":
        scale = (res.abs().amax(dim=(1, 2)) / 2.0 ** 14).contiguous()
        res = (res / scale[:, None, None]).half()
    elif dtype == "bf16":
        res = res.bfloat16()
    return res, sigma, m, scale


def _velocities(nx, ny, vmax):
    """The velocity grid, x fastest."""
    gx = np.linspace(-vmax, vmax, nx) if nx > 1 else np.array([0.3 * vmax])
    gy = np.linspace(-vmax, vmax, ny) if ny > 1 else np.array([-0.4 * vmax])
    return np.tile(gx, ny), np.repeat(gy, nx)


def _frame_model(T):
    """Frame times with a downlink gap in mid-sector, and pointing jitter: a
    bounded random walk (the same for every seed: it belongs to the table)."""
    rng = np.random.default_rng(12)
    times = np.arange(T, dtype=np.float64)
    times[T // 2:] += 40.0
    return times, np.clip(np.cumsum(rng.normal(0, 0.04, size=(T, 2)), 0), -0.15, 0.15)


def _psf_bank(vx, vy, T):
    """Shifts and footprints of an elongated, tilted PSF sampled at the
    trajectory's sub-pixel phase, unit sum: it does not factor into axes."""
    t = np.arange(T, dtype=np.float64)
    cx, cy = vx[:, None] * t, vy[:, None] * t
    sx, sy = np.floor(cx + 0.5), np.floor(cy + 0.5)
    d = np.arange(-2, 3)
    dx = d[None, None, None, :] - (cx - sx)[:, :, None, None]
    dy = d[None, None, :, None] - (cy - sy)[:, :, None, None]
    w = np.exp(-(dx * dx / 1.1 + dy * dy / 0.8 - 0.7 * dx * dy))
    return np.stack([sx, sy], -1).astype(np.int32), w / w.sum((2, 3), keepdims=True)


def _table(c):
    vx, vy = _velocities(c["nx"], c["ny"], c["vmax"])
    if c.get("prf") == "custom":
        return mf.prf_table_create_custom(*_psf_bank(vx, vy, c["T"]))
    times, jitter = _frame_model(c["T"]) if c.get("frames") else (None, None)
    return mf.prf_table_create(vx, vy, c["T"], sigma_px=SIGMA_PRF, kind=KINDS[c.get("prf", "gauss")], times=times,
                               jitter=jitter)


def _score_map(H, W, K, seed):
    """A best-score map as a search over K filters leaves it: noise around
    2.5 with a slow gradient, compact sources, masked blobs without a score."""
    g = _gen(seed)
    yy = torch.arange(H, device=DEV, dtype=torch.float32)[:, None] / H
    s = 2.5 + 0.45 * torch.randn((H, W), generator=g, device=DEV) + 0.5 * (yy - 0.5)
    n = max(1, min(200, H * W // 400))
    peak = torch.zeros((H, W), device=DEV)
    at = torch.randint(0, H * W, (n,), generator=g, device=DEV)
    peak.view(-1)[at] = 2 + 10 * torch.rand((n,), generator=g, device=DEV)
    d = torch.arange(-2, 3, device=DEV, dtype=torch.float32)
    k = torch.exp(-(d[:, None] ** 2 + d ** 2) / 1.5)
    s = s + sum(torch.roll(peak, (i - 2, j - 2), (0, 1)) * float(k[i, j]) for i in range(5) for j in range(5))
    a = torch.randint(0, K, (H, W), generator=g, device=DEV, dtype=torch.int32)
    m = _mask(H, W, 0.01, g).bool()
    return s.masked_fill(m, 0.0).contiguous(), a.masked_fill(m, -1).contiguous()


def _raw_frames(T, H, W, n, seed):
    """Raw frames for the background fit: drifting scattered light (also
    sampled on an n x n grid), a background with jitter terms, noise, rare
    bright outliers."""
    c = synth.background_case_gpu(T=T, H=H, W=W, seed=seed, n=n, device=DEV)
    return c["D"], c["S"], c["jitter"]


def _batch_items(c):
    """The cutouts of a batch: sides, frames, trajectories and types."""
    rng = np.random.default_rng([c["items"], c["side_hi"], c["t_hi"], c["k_hi"]])
    out = []
    for i in range(c["items"]):
        H, W = (int(rng.integers(c["side_lo"], c["side_hi"] + 1)) for _ in range(2))
        K = int(rng.integers(c["k_lo"], c["k_hi"] + 1))
        nx = max(1, int(round(math.sqrt(K))))
        out.append(dict(op="search", T=int(rng.integers(c["t_lo"], c["t_hi"] + 1)), H=H, W=W, nx=nx,
                        ny=max(1, K // nx), vmax=0.1, dtype=["f32", "bf16", "fp16"][i % 3], prf="gauss", mask=0.01,
                        frames=False, cube=False))
    return out


def prepare(case, seed):
    op = case["op"]
    s = {"op": op, "case": case}
    if op == "search":
        s["stack"], s["sigma"], s["mask"], s["scale"] = _sky(case["T"], case["H"], case["W"], case["mask"],
                                                             case["dtype"], seed)
        s["table"] = _table(case)
        s["ws"] = torch.empty(mf.search_workspace_size(s["stack"].shape, s["table"], s["stack"].dtype),
                              dtype=torch.uint8, device=DEV)
    elif op == "rescore":
        s["stack"], s["sigma"], s["mask"], _ = _sky(case["T"], case["H"], case["W"], case["mask"], "f32", seed)
        s["table"] = _table(case)
        s["smax"], s["amax"] = _score_map(case["H"], case["W"], case["nx"] * case["ny"], seed + 77)
        s["ws"] = torch.empty(mf.rescore_workspace_size(case["H"], case["W"], case["k_top"]), dtype=torch.uint8,
                              device=DEV)
    elif op == "detect":
        s["smax"], s["amax"] = _score_map(case["H"], case["W"], 100, seed)
        s["z"] = torch.empty_like(s["smax"]) if case["zmap"] else None
        s["ws"] = torch.empty(mf.detect_workspace_size(case["H"], case["W"], case["max_out"]), dtype=torch.uint8,
                              device=DEV)
    elif op == "refit":
        s["D"], s["S"], s["jitter"] = _raw_frames(case["T"], case["H"], case["W"], case["n"], seed)
        s["R"] = torch.empty_like(s["D"])
        s["ws"] = torch.empty(mf.refit_workspace_size(case["T"]), dtype=torch.uint8, device=DEV)
    else:
        s["batch"] = mf.Batch()
        for i, it in enumerate(_batch_items(case)):
            stack, sigma, mask, scale = _sky(it["T"], it["H"], it["W"], it["mask"], it["dtype"], 100 * seed + i)
            s["batch"].add(stack, sigma, _table(it), mask=mask, frame_scale=scale)
        s["batch"].prepare(device=DEV)
    return s


def _candidates(raw, n):
    """The fields of candidate records, by type."""
    i, f, d = raw.view(torch.int32), raw.view(torch.float32), raw.view(torch.float64)
    return {"yxk": i[:, :3], "snr": d[:, 2], "flux": d[:, 3], "snr_search": f[:, 8], "n": n}


def _detections(raw, n):
    """The fields of detection records, by type."""
    i, f, d = raw.view(torch.int32), raw.view(torch.float32), raw.view(torch.float64)
    return {"yxk_npix": i[:, :4], "z": d[:, 2], "mean": d[:, 3], "sigma": d[:, 4], "snr": f[:, 10], "n": n}


def run(state):
    op, c = state["op"], state["case"]
    if op == "search":
        smax, amax, cube = mf.search(state["stack"], state["sigma"], state["table"], mask=state["mask"],
                                     frame_scale=state["scale"], want_all=c["cube"], workspace=state["ws"])
        return {"snr_max": smax, "argmax": amax, "snr_all": cube}
    if op == "rescore":
        return _candidates(*mf.rescore_topk(state["stack"], state["sigma"], state["table"], state["smax"],
                                            state["amax"], c["k_top"], mask=state["mask"], workspace=state["ws"]))
    if op == "detect":
        raw, n = mf.detect(state["smax"], state["amax"], window=c["window"], threshold=3.0, max_out=c["max_out"],
                           z_out=state["z"], workspace=state["ws"])
        return dict(_detections(raw, n), zmap=state["z"])
    if op == "refit":
        resid, coef = mf.background_refit(state["D"], state["jitter"], c["delta"], c["iterations"],
                                          scatter=state["S"], resid=state["R"], workspace=state["ws"])
        return {"resid": resid, "coef": coef}
    state["batch"].run()
    return [{"snr_max": o[0], "argmax": o[1]} for o in state["batch"].outputs]


# ------------------------------------------------------------------ work ---

def _search_work(c):
    P, K = c["H"] * c["W"], c["nx"] * c["ny"]
    units = P * K * c["T"]
    vx, vy = _velocities(c["nx"], c["ny"], c["vmax"])
    taps = {"gauss": 5, "shiftstack": 1, "custom": 25}[c["prf"]]
    # numerator: the taps of one axis per unit and, once per velocity column,
    # the other axis (factored footprints), or all 25; denominator: one
    # multiply-add per pixel that the trajectory's footprint passes over
    path = np.abs(vx).sum() + np.abs(vy).sum()
    swath = 25 * K + 5 * c["T"] * path if taps > 1 else K + c["T"] * path
    flops = 2.0 * taps * units + (2.0 * taps * P * c["T"] * len(set(vx)) if taps == 5 else 0) + 2.0 * swath * P
    size = 4 if c["dtype"] == "f32" else 2
    return {"bytes": P * (size * c["T"] + 4 + (1 if c["mask"] else 0) + 8 + (4 * K if c["cube"] else 0)),
            "flops": flops}


def work(case):
    op = case["op"]
    if op == "search":
        return _search_work(case)
    if op == "batch":
        w = [_search_work(it) for it in _batch_items(case)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    P = case["H"] * case["W"]
    if op == "rescore":
        taps = case["k_top"] * case["T"] * 25
        return {"bytes": 13 * P + 4 * taps + 40 * case["k_top"], "flops": 6.0 * taps}
    if op == "detect":
        return {"bytes": (12 if case["zmap"] else 8) * P + 56 * case["max_out"], "flops": 20.0 * P}
    return {"bytes": P * (8 * case["T"] + 24), "flops": 26.0 * P * case["T"] * (case["iterations"] + 1)}


# ----------------------------------------------------------------- exact ---

def _axis(kind, ph):
    """Unit-sum 5-pixel profile of one axis at sub-pixel phases ph [...], in
    FP64: the Gaussian integrated over each pixel, or the base pixel alone."""
    d = np.arange(-2, 3)
    if kind == 2:
        return np.broadcast_to((d == 0).astype(np.float64), ph.shape + (5,))
    erf = np.vectorize(math.erf, otypes=[np.float64])
    s = SIGMA_PRF * math.sqrt(2.0)
    g = 0.5 * (erf((d + 0.5 - ph[..., None]) / s) - erf((d - 0.5 - ph[..., None]) / s))
    return g / g.sum(-1, keepdims=True)


def _bank(c):
    """Shifts [K, T, 2] and either axis factors (ux, uy) [K, T, 5] or
    footprints [K, T, 5, 5]."""
    vx, vy = _velocities(c["nx"], c["ny"], c["vmax"])
    if c.get("prf") == "custom":
        sh, w = _psf_bank(vx, vy, c["T"])
        return sh, None, None, w
    times, jit = _frame_model(c["T"]) if c.get("frames") else (np.arange(c["T"], dtype=np.float64),
                                                              np.zeros((c["T"], 2)))
    cx, cy = vx[:, None] * times + jit[:, 0], vy[:, None] * times + jit[:, 1]
    sx, sy = np.floor(cx + 0.5), np.floor(cy + 0.5)
    kind = KINDS[c.get("prf", "gauss")]
    return np.stack([sx, sy], -1).astype(np.int64), _axis(kind, cx - sx), _axis(kind, cy - sy), None


def _inverse_variance(sigma, mask):
    lam = 1.0 / sigma.double() ** 2
    return lam if mask is None else lam.masked_fill(mask.bool(), 0.0)


def _search_seconds(c):
    """About what exact() of a search takes: small launches over the image."""
    n = c["nx"] * c["ny"] * c["T"] * {"gauss": 5, "shiftstack": 1, "custom": 25}[c["prf"]]
    return n * max(5e-6, 24 * c["H"] * c["W"] / 4e12) + c["T"] * c["nx"] * 3e-5


def _exact_search(c, seed):
    stack, sigma, mask, scale = _sky(c["T"], c["H"], c["W"], c["mask"], c["dtype"], seed)
    H, W, T = c["H"], c["W"], c["T"]
    sh, ux, uy, w = _bank(c)
    K = sh.shape[0]
    M = int(np.abs(sh).max()) + 2
    lam = torch.nn.functional.pad(_inverse_variance(sigma, mask), (M, M, M, M))
    N = torch.zeros((K, H, W), dtype=torch.float64, device=DEV)
    D = torch.zeros_like(N)
    cls = {}
    for k in range(K):
        cls.setdefault(sh[k, :, 0].tobytes() + (ux[k].tobytes() if ux is not None else b"%d" % k), []).append(k)
    only = uy is not None and c["prf"] == "shiftstack"
    for t in range(T):
        y = torch.nn.functional.pad(stack[t].double() * (float(scale[t]) if scale is not None else 1.0),
                                    (M, M, M, M)) * lam
        for ks in cls.values():
            x0 = M + int(sh[ks[0], t, 0])
            if w is not None:
                y0 = M + int(sh[ks[0], t, 1])
                for b in range(5):
                    for a in range(5):
                        N[ks[0]].add_(y[y0 + b - 2:y0 + b - 2 + H, x0 + a - 2:x0 + a - 2 + W],
                                      alpha=float(w[ks[0], t, b, a]))
                continue
            h = y[:, x0:x0 + W] if only else sum(y[:, x0 + a - 2:x0 + a - 2 + W] * float(ux[ks[0], t, a])
                                                 for a in range(5))
            for k in ks:
                y0 = M + int(sh[k, t, 1])
                for b in ((2,) if only else range(5)):
                    N[k].add_(h[y0 + b - 2:y0 + b - 2 + H], alpha=float(uy[k, t, b]))
    for k in range(K):  # the inverse variance is the same in every frame: one weight per offset
        G = np.zeros((2 * M + 1, 2 * M + 1))
        f = w[k] if w is not None else uy[k][:, :, None] * ux[k][:, None, :]
        for b in range(5):
            for a in range(5):
                np.add.at(G, (sh[k, :, 1] + b - 2 + M, sh[k, :, 0] + a - 2 + M), f[:, b, a] ** 2)
        for b, a in np.argwhere(G > 0):
            D[k].add_(lam[b:b + H, a:a + W], alpha=float(G[b, a]))
    snr = torch.where(D > 0, N / D.sqrt(), torch.zeros_like(N))
    best = torch.where(D > 0, snr, torch.full_like(snr, -math.inf)).amax(0)
    best = torch.where(torch.isinf(best), torch.zeros_like(best), best)
    return {"snr_max": best, "argmax": None, "snr_all": snr if c["cube"] else None}


def _exact_rescore(c, seed):
    stack, sigma, mask, _ = _sky(c["T"], c["H"], c["W"], c["mask"], "f32", seed)
    smax, amax = _score_map(c["H"], c["W"], c["nx"] * c["ny"], seed + 77)
    H, W = c["H"], c["W"]
    sh, ux, uy, _ = _bank(c)
    lam = _inverse_variance(sigma, mask)
    score = smax.double().masked_fill(amax < 0, -math.inf).view(-1)
    order = torch.sort(score, descending=True, stable=True)[1][:c["k_top"]]
    n = int(min(c["k_top"], int((amax >= 0).sum())))
    order = order[:n]
    k = amax.view(-1)[order].long()
    py, px = order // W, order % W
    sht, uxt, uyt = (torch.from_numpy(np.ascontiguousarray(v)).to(DEV) for v in (sh, ux, uy))
    N = torch.zeros(n, dtype=torch.float64, device=DEV)
    D = torch.zeros_like(N)
    for t in range(c["T"]):
        for b in range(5):
            for a in range(5):
                qy, qx = py + sht[k, t, 1] + b - 2, px + sht[k, t, 0] + a - 2
                ok = (qy >= 0) & (qy < H) & (qx >= 0) & (qx < W)
                qy, qx = qy.clamp(0, H - 1), qx.clamp(0, W - 1)
                wl = uyt[k, t, b] * uxt[k, t, a]
                la = torch.where(ok, lam[qy, qx], torch.zeros_like(N))
                N += wl * la * stack[t][qy, qx].double()
                D += wl * wl * la
    out = {"snr": torch.zeros(c["k_top"], dtype=torch.float64, device=DEV)}
    out["flux"] = torch.zeros_like(out["snr"])
    out["snr"][:n] = torch.where(D > 0, N / D.sqrt(), torch.zeros_like(N))
    out["flux"][:n] = torch.where(D > 0, N / D, torch.zeros_like(N))
    return dict(out, yxk=None, snr_search=None, n=None)


def _box(v, R):
    """Sums over the (2R + 1)^2 square clipped to the image, one axis at a
    time, each window summed by doubling (no long running sums)."""
    for axis in (0, 1):
        n = v.shape[axis]
        p = torch.nn.functional.pad(v.movedim(axis, 0), (0, 0, R, R))
        need, at, acc, width, cur = 2 * R + 1, 0, 0, 1, p
        while need:
            if need & 1:
                acc = acc + cur[at:at + n]
                at += width
            need >>= 1
            cur = cur[:-width] + cur[width:] if need else cur
            width *= 2
        v = acc.movedim(0, axis).contiguous()
    return v


def _exact_detect(c, seed):
    smax, amax = _score_map(c["H"], c["W"], 100, seed)
    H, W, R = c["H"], c["W"], c["window"] // 2
    valid = amax >= 0
    s = torch.where(valid, smax.double(), torch.zeros((), dtype=torch.float64, device=DEV))
    n, s1, s2 = _box(valid.double(), R), _box(s, R), _box(s * s, R)
    mean = s1 / n.clamp(min=1)
    var = (s2 / n.clamp(min=1) - mean * mean).clamp(min=0)
    ok = valid & (n >= 2) & (var > 1e-12 * (mean * mean + var))
    z = torch.where(ok, (smax.double() - mean) / var.sqrt().clamp(min=1e-300), torch.zeros_like(mean))
    flag = ok & (z > 3.0)
    # components: the smallest index spreads over touching candidates
    lab = torch.where(flag, torch.arange(H * W, device=DEV, dtype=torch.float64).view(H, W) - H * W,
                      torch.zeros_like(z))
    while True:
        nxt = torch.where(flag, -torch.nn.functional.max_pool2d(-lab[None, None], 3, 1, 1)[0, 0], lab)
        if torch.equal(nxt, lab):
            break
        lab = nxt
    at = flag.view(-1).nonzero()[:, 0]
    lb, zf = lab.view(-1)[at], z.view(-1)[at]
    by_z = torch.sort(zf, descending=True, stable=True)[1]  # index order among equal z
    by = by_z[torch.sort(lb[by_z], stable=True)[1]]
    first = torch.ones(len(by), dtype=torch.bool, device=DEV)
    first[1:] = lb[by][1:] != lb[by][:-1]
    peaks = torch.sort(at[by[first]])[0]
    peaks = peaks[torch.sort(z.view(-1)[peaks].float(), descending=True, stable=True)[1]][:c["max_out"]]
    out = {}
    for name, v in (("z", z), ("mean", mean), ("sigma", var.sqrt())):
        out[name] = torch.zeros(max(c["max_out"], 1), dtype=torch.float64, device=DEV)
        out[name][:len(peaks)] = v.view(-1)[peaks]
    return dict(out, yxk_npix=None, snr=None, n=None, zmap=z if c["zmap"] else None)


def _exact_refit(c, seed):
    D, S, jit = _raw_frames(c["T"], c["H"], c["W"], c["n"], seed)
    T, H, W, n = c["T"], c["H"], c["W"], c["n"]
    x, y = torch.from_numpy(jit).to(DEV).T
    phi = torch.stack([torch.ones_like(x), x, y, x * x, y * y, x * y], 1)
    Q, Rm = torch.linalg.qr(phi)

    def axis(size):  # pixel centres on the scattered-light grid, clamped at its edge
        u = ((torch.arange(size, device=DEV, dtype=torch.float64) + 0.5) * n / size - 0.5).clamp(0, n - 1)
        i0 = u.floor().long()
        return i0, (i0 + 1).clamp(max=n - 1), u - i0
    i0, i1, fy = axis(H)
    j0, j1, fx = axis(W)
    resid = torch.empty((T, H, W), dtype=torch.float64, device=DEV)
    coef = torch.empty((H, W, 6), dtype=torch.float64, device=DEV)
    rows = max(1, int(2e8 // (T * W)))
    for r in range(0, H, rows):
        e = min(H, r + rows)
        St = S.double()
        top = St[:, i0[r:e]][:, :, j0] * (1 - fx) + St[:, i0[r:e]][:, :, j1] * fx
        bot = St[:, i1[r:e]][:, :, j0] * (1 - fx) + St[:, i1[r:e]][:, :, j1] * fx
        v = (D[:, r:e].double() - (top * (1 - fy[r:e, None]) + bot * fy[r:e, None])).reshape(T, -1)
        del top, bot
        beta = Q.T @ v
        for _ in range(c["iterations"]):
            beta = beta + Q.T @ (v - Q @ beta).clamp(-c["delta"], c["delta"])
        resid[:, r:e] = (v - Q @ beta).view(T, e - r, W)
        coef[r:e] = torch.linalg.solve_triangular(Rm, beta, upper=True).T.reshape(e - r, W, 6)
    return {"resid": resid, "coef": coef}


def exact(case, seed):
    """What run() returns, in FP64 from the definition; None where that takes
    too long or an output has no such value (indices and counts)."""
    op = case["op"]
    if op == "search":
        return _exact_search(case, seed) if _search_seconds(case) < 15 else None
    if op == "rescore":
        return _exact_rescore(case, seed) if case["T"] * 25 * 4e-4 < 15 else None
    if op == "detect":
        return _exact_detect(case, seed)
    if op == "refit":
        return _exact_refit(case, seed)
    items = _batch_items(case)
    if sum(_search_seconds(it) for it in items) > 15:
        return None
    return [{k: v for k, v in _exact_search(it, 100 * seed + i).items() if k != "snr_all"}
            for i, it in enumerate(items)]
