"""Performance cases: the imaging work a user of this library has it do, through its public entry points.

Every case images synthetic scans of the repository's shared radar (77 GHz, 4 GHz over 40 us, 0.25 m arm): point
targets, receiver noise and, where the path takes them, rotation errors.  A case's `path` names the entry points:

  image      rosar.image: range compression, then the sparse azimuth filter tap by tap (any pulse count)
  image_fft  rosar.image_fft: the same with the frequency-domain plan of a weight design
  scans      rosar.image_fft_scans: a sequence of scans of one design
  batch      rosar.Batch: scans of uneven sizes bound to one graph launch
  migrating  rosar.image_migrating_fft: taps that follow the pulses' peak bins
  bpa        rosar.range_compress, then rosar.bpa (nominal positions, or supplied rotation errors)
  sas_time   rosar.sas_time or sas_time_planned: Algorithm 2 on the raw cube
  bpa_time   rosar.bpa_time or bpa_time_planned: Eq. (14) on the raw cube
  diff       one autofocus step: image, loss against a reference image, gradients of weights, phases and raw cube
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2309_08038_gb300 as rosar
from paper_2309_08038_gb300 import autograd as rosar_grad

C = 299792458.0
FC, SLOPE, T_ADC, T_START, R0 = 77e9, 1e14, 24e-6, 8e-6, 0.25      # the radar of every configuration here
DR = C / (2.0 * SLOPE * T_ADC)                                     # range bin, the same for every L
SMOOTH = sorted(2 ** a * 3 ** b * 5 ** c for a in range(15) for b in range(10) for c in range(7)
                if 360 <= 2 ** a * 3 ** b * 5 ** c <= 14400)       # pulse counts with a frequency-domain plan


def listed():
    return [
        # the tiny scan (360 x 64, 16 taps): one call of a few microseconds, launches and host time count
        {"name": "image_tiny", "path": "image", "n_az": 360, "L": 64, "K": 16, "per_row": False},
        # a free-running turntable: an indoor-sized scan whose pulse count is a prime, so no plan exists for it
        {"name": "image_prime", "path": "image", "n_az": 3607, "L": 256, "K": 64, "per_row": False},
        # the paper's rotation (800 pulses, 225 samples padded to 256), one scan per call
        {"name": "fft_800", "path": "image_fft", "n_az": 800, "L": 256, "K": 64, "per_row": False},
        # the high-resolution scan (14400 x 1024, per-row taps)
        {"name": "fft_highres", "path": "image_fft", "n_az": 14400, "L": 1024, "K": 128, "per_row": True},
        # a stream of indoor scans of one weight design
        {"name": "scans_indoor", "path": "scans", "n_scans": 16, "n_az": 3600, "L": 256, "K": 64},
        # a quarter of the batched workload: 64 scans of uneven sizes in one launch
        {"name": "batch_64", "path": "batch", "n_scans": 64, "pulses": "1800,3600,7200", "samples": "128,256,512,1024",
         "mix": 3, "plan": True},
        # the indoor scan with every tap reading its pulse's peak bin
        {"name": "migrating_indoor", "path": "migrating", "n_az": 3600, "L": 256, "K": 64},
        # FFT+BPA of the indoor scan, the comparison image: nominal positions, and with the rotation errors supplied
        {"name": "bpa_nominal", "path": "bpa", "n_az": 3600, "L": 256, "M": 600, "errors": False},
        {"name": "bpa_errors", "path": "bpa", "n_az": 3600, "L": 256, "M": 600, "errors": True},
        # the paper's SAS on the raw cube, weights new with each call
        {"name": "sas_time_indoor", "path": "sas_time", "n_az": 3600, "L": 256, "K": 64, "planned": False},
        # the paper's BPA on the raw cube of a radar whose plan is kept
        {"name": "bpa_time_plan", "path": "bpa_time", "n_az": 3600, "L": 256, "M": 600, "planned": True},
        # autofocus of 16 indoor scans that share their weights
        {"name": "diff_16", "path": "diff", "n_scans": 16, "n_az": 3600, "L": 256, "K": 64, "raw_grad": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _smooth(rng, lo, hi):
    at = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min((n for n in SMOOTH if lo <= n <= hi), key=lambda n: (abs(math.log(n / at)), n))


def draw(rng):
    """One more case: the paths by how often a program takes them, the sizes spread over the logarithm of their range."""
    path = rng.choices(["image", "image_fft", "scans", "batch", "migrating", "bpa", "sas_time", "bpa_time", "diff"],
                       [4, 5, 4, 3, 2, 3, 1, 1, 2])[0]
    while True:
        L = 2 ** rng.randint(6, 10)
        K = _log_int(rng, 16, 128)
        if path == "image":
            c = {"n_az": _log_int(rng, 360, 7200), "L": L, "K": K, "per_row": rng.random() < 0.3}
            fits = c["n_az"] * L <= 8e6
        elif path == "image_fft":
            c = {"n_az": _smooth(rng, 360, 14400), "L": L, "K": K, "per_row": rng.random() < 0.3}
            fits = c["n_az"] * L <= 14400 * 1024
        elif path == "scans":
            c = {"n_scans": rng.randint(2, 24), "n_az": _smooth(rng, 360, 7200), "L": L, "K": K}
            fits = c["n_scans"] * c["n_az"] * L <= 3e7
        elif path == "batch":
            pulses = [_smooth(rng, 360, 7200) for _ in range(3)] if rng.random() < 0.5 else [1800, 3600, 7200]
            c = {"n_scans": _log_int(rng, 6, 64), "pulses": ",".join(map(str, pulses)), "samples": "64,128,256,512",
                 "mix": rng.randrange(1000), "plan": rng.random() < 0.8}
            fits = c["plan"] or c["n_scans"] <= 16
        elif path == "migrating":
            c = {"n_az": _smooth(rng, 360, 7200), "L": L, "K": K}
            fits = c["n_az"] * L <= 4e6
        elif path == "bpa":
            n = _log_int(rng, 360, 7200)
            c = {"n_az": n, "L": min(L, 512), "M": max(2, int(n * rng.uniform(0.1, 0.2))), "errors": rng.random() < 0.5}
            fits = c["n_az"] * c["L"] * c["M"] <= 8e8
        elif path in ("sas_time", "bpa_time"):
            n = _log_int(rng, 360, 4500)
            taps = {"K": K} if path == "sas_time" else {"M": max(2, int(n * rng.uniform(0.1, 0.17)))}
            c = {"n_az": n, "L": 16 * rng.randint(4, 20), **taps, "planned": rng.random() < 0.5}
            fits = n * c["L"] ** 2 * list(taps.values())[0] <= (1.4e11 if c["planned"] else 8e10)
        else:
            c = {"n_scans": rng.randint(2, 16), "n_az": _smooth(rng, 360, 7200), "L": min(L, 512), "K": K,
                 "raw_grad": rng.random() < 0.5}
            fits = c["n_scans"] * c["n_az"] * c["L"] <= 1.5e7
        if fits:
            return {"path": path, **c}


# ------------------------------------------------------------------------------------------------ inputs --

def _radar(L):
    return rosar.Radar(FC, SLOPE, T_ADC / L, T_START, R0, C)


def _k_mid(L):
    return 2.0 * math.pi * (FC + SLOPE * (T_START + (T_ADC / L) * (L - 1) / 2.0)) / C


def _window(L, device):
    m = torch.arange(L, dtype=torch.float64, device=device)
    return (0.5 - 0.5 * torch.cos(2.0 * math.pi * m / (L - 1))).float()


def _scan(gen, n_az, L, dphi=None, dr=None, targets=8, out=None):
    """Raw cube [n_az, L] complex64: Rayleigh targets seen by the rotating antenna, and noise 20 dB below one."""
    dev = gen.device
    f8 = dict(dtype=torch.float64, device=dev)
    R = R0 + DR + torch.rand(targets, generator=gen, **f8) * (0.9 * L - 2) * DR
    ang = torch.rand(targets, generator=gen, **f8) * (2.0 * math.pi)
    amp = torch.randn(targets, 2, generator=gen, **f8)
    ph = torch.arange(n_az, **f8) * (2.0 * math.pi / n_az) + (0.0 if dphi is None else dphi.double())
    rr = torch.full((n_az,), R0, **f8) + (0.0 if dr is None else dr.double())
    raw = torch.randn(n_az, L, 2, generator=gen, dtype=torch.float32, device=dev).mul_(math.sqrt(0.005))
    t = T_START + torch.arange(L, **f8) * (T_ADC / L)
    for q in range(targets):
        Rn = torch.sqrt(R[q] ** 2 + rr ** 2 - 2.0 * R[q] * rr * torch.cos(ang[q] - ph))
        p = ((R[q] * torch.cos(ang[q] - ph) - rr) / Rn).clamp_min(0.0)
        turns = (2.0 / C) * Rn[:, None] * (FC + SLOPE * t)[None, :]
        x = (2.0 * math.pi * (turns - torch.floor(turns))).float()
        s, c = torch.sin(x), torch.cos(x)
        a, b = (amp[q, 0] * p).float()[:, None], (amp[q, 1] * p).float()[:, None]
        raw[..., 0] += a * c - b * s
        raw[..., 1] += a * s + b * c
    raw = torch.view_as_complex(raw)
    if out is not None:
        return out.copy_(raw)
    return raw


def _design(rs, n_az, L, K, per_row, device):
    """Sparse taps in an aperture of a sixth of the turn and their weights: the conjugate steering vector at the taps
    under a raised-cosine taper, rows of unit norm; and every tap's row offset to its peak bin."""
    M = max(K, n_az // 6)
    draws = [np.sort(rs.choice(M, K, replace=False)) - M // 2 for _ in range(L if per_row else 1)]
    o = torch.from_numpy(np.stack(draws).astype(np.int32)).to(device)
    f8 = dict(dtype=torch.float64, device=device)
    R = R0 + torch.arange(L, **f8)[:, None] * DR
    cosd = torch.cos(o.double() * (2.0 * math.pi / n_az))
    rho = torch.sqrt((R * R + R0 * R0 - 2.0 * R * R0 * cosd).clamp_min(0.0))
    p = torch.where(rho > 0, (R * cosd - R0).clamp_min(0.0) / rho.clamp_min(1e-9), torch.ones_like(rho))
    v = (0.55 + 0.45 * torch.cos(o.double() * (2.0 * math.pi / M))) * p
    v = torch.polar(v, -2.0 * _k_mid(L) * rho)
    w = (v / torch.linalg.vector_norm(v, dim=1, keepdim=True).clamp_min(1e-30)).to(torch.complex64)
    dl = (torch.floor(rho / DR + 0.5) - torch.arange(L, **f8)[:, None]).to(torch.int32).expand(L, K).contiguous()
    return (o if per_row else o[0].contiguous()), w, dl


def _batch_shapes(case):
    rs = np.random.RandomState(7 + case["mix"])
    n = rs.choice([int(x) for x in case["pulses"].split(",")], case["n_scans"])
    L = rs.choice([int(x) for x in case["samples"].split(",")], case["n_scans"])
    K = rs.choice([32, 64, 128], case["n_scans"])
    return [(int(a), int(b), int(min(c, a // 6))) for a, b, c in zip(n, L, K)]


def _inputs(case, seed):
    """The tensors of a case, without anything of the library's."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    rs = np.random.default_rng(seed)
    path = case["path"]
    if path == "batch":
        shapes = _batch_shapes(case)
        flat = torch.empty(sum(n * L for n, L, _ in shapes), dtype=torch.complex64, device=dev)
        scans, at = [], 0
        for n_az, L, K in shapes:
            raw = _scan(gen, n_az, L, targets=4, out=flat[at:at + n_az * L].view(n_az, L))
            o, w, _ = _design(rs, n_az, L, K, False, dev)
            scans.append({"raw": raw, "w": w, "o": o, "win": _window(L, dev)})
            at += n_az * L
        return {"scans": scans, "total": at}
    n_az, L = case["n_az"], case["L"]
    d = {"win": _window(L, dev)}
    if "K" in case:
        d["o"], d["w"], d["dl"] = _design(rs, n_az, L, case["K"], case.get("per_row", False), dev)
    if case.get("errors"):
        d["dphi"] = torch.randn(n_az, generator=gen, device=dev) * math.radians(0.05)
        d["dr"] = torch.randn(n_az, generator=gen, device=dev) * 1e-3
    if "n_scans" in case:
        d["raw"] = torch.empty(case["n_scans"], n_az, L, dtype=torch.complex64, device=dev)
        for s in range(case["n_scans"]):
            _scan(gen, n_az, L, out=d["raw"][s])
    else:
        d["raw"] = _scan(gen, n_az, L, d.get("dphi"), d.get("dr"))
    if path == "diff":
        # the reference image is that of the error-free scans; the phase errors are half corrected already
        d["ref"] = torch.stack([_image64(r, d["win"], d["w"], d["o"]).to(torch.complex64) for r in d["raw"]])
        err = torch.randn(case["n_scans"], n_az, generator=gen, device=dev) * 0.3
        d["raw"] = d["raw"] * torch.polar(torch.ones_like(err), err)[:, :, None]
        d["eps"] = -0.5 * err
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    path = case["path"]
    d["path"] = path
    if path == "batch":
        d["S"] = torch.empty(d["total"], dtype=torch.complex64, device="cuda")
        d["out"] = torch.empty_like(d["S"])
        at = 0
        for sc in d["scans"]:
            n_az, L = sc["raw"].shape
            sc["S"], sc["out"] = (d[x][at:at + n_az * L].view(L, n_az) for x in ("S", "out"))
            at += n_az * L
            if case["plan"]:
                sc["H"] = rosar.azimuth_plan(sc["w"], sc["o"], n_az)
        d["batch"] = rosar.Batch(d["scans"])
        return d
    n_az, L = case["n_az"], case["L"]
    radar = d["radar"] = _radar(L)
    if path in ("image_fft", "scans"):
        d["H"] = rosar.azimuth_plan(d["w"], d["o"], n_az)
    elif path == "migrating":
        d["plan"] = rosar.azimuth_plan_migrating(d["w"], d["o"], d["dl"], n_az)
    elif path == "bpa":
        d["M"] = case["M"]
    elif path == "sas_time":
        d["plan"] = rosar.sas_time_plan(d["win"], d["w"], d["o"], radar, n_az, L) if case["planned"] else None
    elif path == "bpa_time":
        d["M"] = case["M"]
        d["plan"] = rosar.bpa_time_plan(d["win"], radar, n_az, L, L, case["M"]) if case["planned"] else None
    elif path == "diff":
        d["w"].requires_grad_(True)
        d["eps"].requires_grad_(True)
        d["raw"].requires_grad_(case["raw_grad"])
    if path in ("image_fft", "scans"):       # a program that images scan after scan keeps its scratch and image
        lead = (case["n_scans"],) if path == "scans" else ()
        d["ws"] = torch.empty((2, L, n_az) if lead else (L, n_az), dtype=torch.complex64, device="cuda")
        d["out"] = torch.empty((*lead, L, n_az), dtype=torch.complex64, device="cuda")
    return d


def run(d):
    path = d["path"]
    if path == "image":
        return rosar.image(d["raw"], d["win"], d["w"], d["o"])
    if path == "image_fft":
        return rosar.image_fft(d["raw"], d["win"], d["H"], workspace=d["ws"], out=d["out"])
    if path == "scans":
        return rosar.image_fft_scans(d["raw"], d["win"], d["H"], workspace=d["ws"], out=d["out"])
    if path == "batch":
        d["batch"].launch()
        return d["out"]
    if path == "migrating":
        return rosar.image_migrating_fft(d["raw"], d["win"], d["plan"])
    if path == "bpa":
        S = rosar.range_compress(d["raw"], d["win"])
        return rosar.bpa(S, d["radar"], S.shape[0], d["M"], dphi=d.get("dphi"), dr=d.get("dr"))
    if path == "sas_time":
        if d["plan"] is not None:
            return rosar.sas_time_planned(d["raw"], d["plan"])
        return rosar.sas_time(d["raw"], d["win"], d["w"], d["o"], d["radar"])
    if path == "bpa_time":
        if d["plan"] is not None:
            return rosar.bpa_time_planned(d["raw"], d["plan"])
        return rosar.bpa_time(d["raw"], d["win"], d["radar"], d["raw"].shape[1], d["M"])
    S = rosar_grad.range_compress(d["raw"], d["win"])
    img = rosar_grad.sparse_azimuth_phase(S, d["eps"], d["w"], d["o"])
    loss = rosar_grad.image_l2_loss(img, d["ref"])
    wanted = [d["w"], d["eps"]] + ([d["raw"]] if d["raw"].requires_grad else [])
    return {"loss": loss.detach(), "grads": torch.autograd.grad(loss, wanted)}


def work(case):
    """Inputs (the raw cube, the weights or the plan) read once, images or gradients written once; the transforms at
    5 N log2 N, a tap or a pixel's pulse at a complex multiply-add (8) and its geometry, as the path defines them."""
    path = case["path"]
    if path == "batch":
        b = f = 0
        for n, L, K in _batch_shapes(case):
            px = n * L
            b += 16 * px + (8 * px if case["plan"] else 8 * L * K + 4 * K)
            f += px * (5 * math.log2(L) + (10 * math.log2(n) + 6 if case["plan"] else 8 * K))
        return {"bytes": b, "flops": f}
    n, L, K = case["n_az"], case["L"], case.get("K", case.get("M"))
    px, s = n * L, case.get("n_scans", 1)
    taps = 8 * L * K + 4 * K * (L if case.get("per_row") else 1) + 4 * L
    fft, row = 5 * math.log2(L), 10 * math.log2(n) + 6
    if path == "image":
        return {"bytes": 16 * px + taps, "flops": px * (fft + 8 * K)}
    if path in ("image_fft", "scans"):
        return {"bytes": 16 * px * s + 8 * px, "flops": s * px * (fft + row)}
    if path == "migrating":
        return {"bytes": 16 * px + 3 * 8 * px, "flops": px * (fft + row + 16)}
    if path == "bpa":
        return {"bytes": 16 * px + 4 * L + (8 * n if case["errors"] else 0), "flops": px * (fft + (30 if case["errors"] else 12) * K)}
    if path == "sas_time":
        return {"bytes": 16 * px + (16 * L * K * L if case["planned"] else taps), "flops": 8 * px * K * L}
    if path == "bpa_time":
        return {"bytes": 16 * px + (16 * L * K * L if case["planned"] else 4 * L), "flops": 8 * px * K * L}
    # raw and the reference in, the gradients out; two transforms of every row and one inverse of each, twice
    grad = 8 * px * s if case["raw_grad"] else 0
    return {"bytes": 16 * px * s + grad + 16 * L * K + 8 * n * s, "flops": s * px * (2 * fft + 2 * row + 30)}


# ------------------------------------------------------------------------------------------- in 64 bits --

def _compress64(raw, win):
    """Centred range compression [.., n_az, L] -> [.., L, n_az] in complex128."""
    L = raw.shape[-1]
    l = torch.arange(L, dtype=torch.float64, device=raw.device)
    x = math.pi * torch.remainder(l * (L - 1) / L, 2.0)
    c = torch.polar(torch.ones_like(x), x)
    return (torch.fft.fft(raw.to(torch.complex128) * win.double(), dim=-1) * c).transpose(-1, -2)


def _taps64(w, o, n_az, dl=None, d=0):
    """The transform of the row's taps laid out as a circular filter, [L, n_az] complex128."""
    L, K = w.shape
    g = torch.zeros(L, n_az, dtype=torch.complex128, device=w.device)
    w = w.to(torch.complex128) if dl is None else w.to(torch.complex128) * (dl == d)
    at = torch.remainder(-o.long(), n_az).expand(L, K)
    return torch.fft.fft(g.scatter_add(1, at, w), dim=-1)


def _image64(raw, win, w, o):
    S = _compress64(raw, win)
    return torch.fft.ifft(torch.fft.fft(S, dim=-1) * _taps64(w, o, raw.shape[-2]), dim=-1)


def _migrating64(d, n_az, L):
    X = torch.fft.fft(_compress64(d["raw"], d["win"]), dim=-1)
    Y = torch.zeros_like(X)
    for q in range(int(d["dl"].min()), int(d["dl"].max()) + 1):
        lo, hi = max(0, -q), min(L, L - q)
        Y[lo:hi] += X[lo + q:hi + q] * _taps64(d["w"], d["o"], n_az, d["dl"], q)[lo:hi]
    return torch.fft.ifft(Y, dim=-1)


def _bpa64(d, n_az, L, M):
    S = _compress64(d["raw"], d["win"])
    S = torch.cat([S, torch.zeros(3, n_az, dtype=S.dtype, device=S.device)])         # bins past the last read zero
    f8 = dict(dtype=torch.float64, device=S.device)
    R = R0 + torch.arange(L, **f8)[:, None] * DR
    eps = d["dphi"].double() if "dphi" in d else torch.zeros(1, **f8)
    rn = R0 + (d["dr"].double() if "dr" in d else torch.zeros(1, **f8))
    out = torch.zeros(L, n_az, dtype=torch.complex128, device=S.device)
    for q in range(-(M // 2), M - M // 2):
        a = 2.0 * math.pi * q / n_az + torch.roll(eps, -q)
        r = torch.roll(rn, -q)
        sh = torch.sin(0.5 * a) ** 2
        Rn = torch.sqrt((R - r) ** 2 + 4.0 * R * r * sh)
        p = torch.where(Rn > 0, ((R - r) - 2.0 * R * sh).clamp_min(0.0) / Rn.clamp_min(1e-300), torch.ones_like(Rn))
        x = Rn / DR
        lo = torch.floor(x).clamp(0, L).long().expand(L, n_az)
        Sq = torch.roll(S, -q, dims=1)
        f = x - torch.floor(x)
        v = (1.0 - f) * torch.gather(Sq, 0, lo) + f * torch.gather(Sq, 0, lo + 1)
        out += torch.polar(p, -2.0 * _k_mid(L) * Rn) * v
    return out


def _time64(d, n_az, L, taps, coef, rho):
    """sum_k coef[r, k] sum_m win[m] exp(-2 pi i tau_k slope t_s (m - mid)) raw[theta + o_k, m], one matrix product a tap."""
    raw = d["raw"].to(torch.complex128) * d["win"].double()
    m = torch.arange(L, dtype=torch.float64, device=raw.device) - (L - 1) / 2.0
    out = torch.zeros(n_az, L, dtype=torch.complex128, device=raw.device)
    for k, o in enumerate(taps):
        turns = (2.0 * rho[:, k] / C * SLOPE * (T_ADC / L))[None, :] * m[:, None]
        ph = -2.0 * math.pi * torch.remainder(turns, 1.0)
        out += torch.roll(raw, -o, dims=0) @ (torch.polar(torch.ones_like(ph), ph) * coef[:, k][None, :])
    return out.T


def _diff64(case, d):
    w = d["w"].to(torch.complex128).requires_grad_(True)
    eps = d["eps"].double().requires_grad_(True)
    raw = d["raw"].to(torch.complex128).requires_grad_(case["raw_grad"])
    S = _compress64(raw, d["win"]) * torch.polar(torch.ones_like(eps), eps)[:, None, :]
    img = torch.fft.ifft(torch.fft.fft(S, dim=-1) * _taps64(w, d["o"], case["n_az"]), dim=-1)
    e = img - d["ref"].to(torch.complex128)
    loss = (e.real ** 2 + e.imag ** 2).sum()
    return {"loss": loss.detach(), "grads": torch.autograd.grad(loss, [w, eps] + ([raw] if case["raw_grad"] else []))}


def exact(case, seed):
    d = _inputs(case, seed)
    path = case["path"]
    if path == "batch":
        out = torch.empty(d["total"], dtype=torch.complex128, device="cuda")
        at = 0
        for sc in d["scans"]:
            n = sc["raw"].numel()
            out[at:at + n] = _image64(sc["raw"], sc["win"], sc["w"], sc["o"]).reshape(-1)
            at += n
        return out
    n_az, L = case["n_az"], case["L"]
    if path in ("image", "image_fft"):
        return _image64(d["raw"], d["win"], d["w"], d["o"])
    if path == "scans":
        return torch.stack([_image64(r, d["win"], d["w"], d["o"]) for r in d["raw"]])
    if path == "migrating":
        return _migrating64(d, n_az, L)
    if path == "bpa":
        return _bpa64(d, n_az, L, case["M"])
    if path == "diff":
        return _diff64(case, d)
    f8 = dict(dtype=torch.float64, device="cuda")
    R = R0 + torch.arange(L, **f8)[:, None] * DR
    taps = d["o"].tolist() if path == "sas_time" else list(range(-(case["M"] // 2), case["M"] - case["M"] // 2))
    sh = torch.sin(torch.tensor(taps, **f8)[None, :] * (math.pi / n_az)) ** 2
    rho = torch.sqrt((R - R0) ** 2 + 4.0 * R * R0 * sh)
    if path == "sas_time":
        return _time64(d, n_az, L, taps, d["w"].to(torch.complex128), rho)
    p = torch.where(rho > 0, ((R - R0) - 2.0 * R * sh).clamp_min(0.0) / rho.clamp_min(1e-300), torch.ones_like(rho))
    return _time64(d, n_az, L, taps, torch.polar(p, -2.0 * _k_mid(L) * rho), rho)
