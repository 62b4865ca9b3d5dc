"""What a user of the framework has it do, as measurable cases: searches of one dedispersed series
in the precisions a pulsar search runs (the paper compares FP32 and BF16), batches of dispersion
trials, the single blocks of the path on their own (long FFT, plane, peak list), and the
refinement of candidates with its gradient.  Sizes are those of the workloads in fdas_synth (the
single chirp, the pulse trains, the batch, the refinement) and of the tests between them; `draw`
spreads over the same ranges, with odd tap counts and template counts.

A case is a dict with a `kind`:
  search    fdas_search on one series: plane, peak list, peak count
  batch     fdas_batch_search over series of uneven length and zmax: peak lists and counts
  spectrum  fdas_spectrum: the long FFT with its normalisation
  plane     fdas_plane from a spectrum, in one of the plane precisions
  peaks     fdas_peaks on a given plane (harmonic sums and the peak list alone)
  refine    refine(): gradient ascent from seeds near injected signals
  interp    interp_power() and its backward pass at candidate points
"""
import math
import random

import numpy as np
import torch

import paper_2206_12205_gb300 as fd
from paper_2206_12205_gb300 import fdas as ft
from paper_2206_12205_gb300 import refine as rf
from paper_2206_12205_gb300.batch import BatchSearch

DEV = "cuda"
# thresholds of the searches: about one noise peak per level on a 2^23-sample, 85-template plane
THR = (40.0, 44.0, 51.0, 64.0, 88.0)
# thresholds of a candidate list that a later sifting step thins out: thousands of noise peaks
THR_LOW = (26.0, 30.0, 38.0, 52.0, 78.0)


def listed():
    return [
        # the smallest search of the workloads: one short series, 17 templates, level 1 only; a
        # call of this size is launches and latency
        dict(name="search_fp32_2e16", kind="search", n=1 << 16, zmax=16, taps=64, seg=1024, prec="fp32", harm=1,
             low=True),
        # a short integration searched through all harmonic levels in BF16
        dict(name="search_bf16_2e18", kind="search", n=1 << 18, zmax=20, taps=64, seg=8192, prec="bf16", harm=16),
        # one ordinary trial of a dedispersed observation (the batch workload's middle zmax)
        dict(name="search_bf16_2e21", kind="search", n=1 << 21, zmax=50, taps=128, seg=8192, prec="bf16", harm=16),
        # the precision workload: 2^23 samples, 85 templates, 256 taps, in BF16 and in FP32
        dict(name="search_bf16_2e23", kind="search", n=1 << 23, zmax=84, taps=256, seg=8192, prec="bf16", harm=16),
        dict(name="search_fp32_2e23", kind="search", n=1 << 23, zmax=84, taps=256, seg=2048, prec="fp32", harm=16),
        # the search variants: median normalisation per block of bins (red noise) and sums anchored
        # at the highest harmonic
        dict(name="search_variants_2e21", kind="search", n=1 << 21, zmax=50, taps=128, seg=8192, prec="bf16", harm=16,
             norm_block=4096, harm_mode=1),
        # many dispersion trials in one call, the way an observation is searched
        dict(name="batch_bf16_12", kind="batch", series=12, log2_lo=21, log2_hi=23, prec="bf16", lanes=3, pick=2),
        # the plane alone in its compensated precision, and by direct correlation of few, short templates
        dict(name="plane_split_2e21", kind="plane", n=1 << 21, zmax=84, taps=256, seg=8192, prec="bf16_split"),
        dict(name="plane_direct_2e22", kind="plane", n=1 << 22, zmax=20, taps=64, seg=8192, prec="bf16_direct"),
        # the peak list of an FP32 plane kept on the device, at a sifting step's low thresholds
        dict(name="peaks_fp32_2e21", kind="peaks", n=1 << 21, zmax=84, prec="fp32", harm=16),
        # sub-bin refinement of a candidate list, and the interpolated power with its gradient
        dict(name="refine_16384", kind="refine", n=1 << 21, taps=256, zmax=84, cands=16384, steps=20),
        dict(name="interp_fp64_4096", kind="interp", n=1 << 21, taps=256, zmax=84, points=4096, fp64=True),
    ]


def _taps(rng, zmax, mult, most=1024):
    """A tap count that holds the widest response (m/2 >= zmax + 12), not only powers of two."""
    m = int(2 * (zmax + 12) * math.exp(rng.uniform(0.0, math.log(1.6))))
    m = max(32, m + (-m) % mult)
    return min(m, most)


def _zmax(rng):
    return 2 * int(round(math.exp(rng.uniform(math.log(4), math.log(42)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "search", "batch", "spectrum", "plane", "plane", "peaks", "refine",
                       "interp"])
    zmax = _zmax(rng)
    log2n = rng.randint(16, 23)
    if kind == "search":
        prec = rng.choice(["bf16", "bf16", "fp32", "fp32", "fp16_scaled", "bf16_direct"])
        mult = 8 if prec == "bf16_direct" else 2
        c = dict(kind=kind, n=1 << log2n, zmax=zmax, taps=_taps(rng, zmax, mult, 240 if mult == 8 else 1024),
                 seg=rng.choice([1024, 2048, 4096, 8192]) if prec == "fp32" else 8192, prec=prec,
                 harm=rng.choice([1, 4, 8, 16, 16]))
        if c["taps"] > c["seg"] // 2:
            c["seg"] = 2048
        if rng.random() < 0.2:
            c["norm_block"] = 1 << rng.randint(8, 13)
        if rng.random() < 0.2:
            c["harm_mode"] = 1
            c["n"] = min(c["n"], 1 << 21)
        return c
    if kind == "batch":
        hi = rng.randint(18, 22)
        return dict(kind=kind, series=rng.randint(3, 16), log2_lo=max(16, hi - rng.randint(0, 3)), log2_hi=hi,
                    prec=rng.choice(["bf16", "bf16", "fp32"]), lanes=rng.randint(1, 4), pick=rng.randint(0, 1 << 20))
    if kind == "spectrum":
        c = dict(kind=kind, n=1 << rng.randint(14, 25))
        if rng.random() < 0.3:
            c["norm_block"] = 1 << rng.randint(8, 13)
        return c
    if kind == "plane":
        prec = rng.choice(["bf16", "bf16_split", "fp32", "fp16_scaled", "bf16_direct", "fp8_direct"])
        mult = {"bf16_direct": 8, "fp8_direct": 16}.get(prec, 2)
        c = dict(kind=kind, n=1 << min(log2n, 22), zmax=zmax, taps=_taps(rng, zmax, mult, 240 if mult > 2 else 1024),
                 seg=rng.choice([2048, 4096, 8192]), prec=prec)
        return c
    if kind == "peaks":
        return dict(kind=kind, n=1 << rng.randint(16, 22), zmax=zmax, prec=rng.choice(["bf16", "fp32"]),
                    harm=rng.choice([2, 8, 16]), harm_mode=int(rng.random() < 0.2))
    size = int(math.exp(rng.uniform(math.log(200), math.log(16000))))
    c = dict(kind=kind, n=1 << rng.randint(18, 22), zmax=zmax, taps=_taps(rng, zmax, 2))
    if kind == "refine":
        c.update(cands=size, steps=rng.randint(5, 20))
    else:
        c.update(points=size, fp64=rng.random() < 0.5)
    return c


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _phase(n, r0, z0, at=0.0):
    u = torch.arange(n, dtype=torch.float64, device=DEV) / n
    c = at + u * (r0 + 0.5 * z0 * u)
    return c - torch.round(c)


def _series(n, zmax, seed, chirps=0, trains=4):
    """Unit Gaussian noise with accelerated signals: `trains` pulse trains (SNR 8-30, 5 % duty,
    several harmonics inside the spectrum) and `chirps` single sinusoids; float32, and the (r, z)
    of each injected harmonic with an expected power of 30 or more."""
    rng = random.Random(int(seed))
    x = torch.randn(n, generator=_gen(seed), device=DEV, dtype=torch.float32)
    truth = []
    w = 0.05 / (2.0 * math.sqrt(2.0 * math.log(2.0)))
    c2 = np.exp(-4.0 * math.pi ** 2 * np.arange(1, 200, dtype=np.float64) ** 2 * w * w)
    share = c2 / c2.sum()
    for _ in range(trains):
        r0 = n / 2 * math.exp(rng.uniform(math.log(0.004), math.log(0.1)))
        z0 = rng.uniform(-0.95, 0.95) * zmax
        snr = rng.uniform(8.0, 30.0)
        s = torch.exp(-0.5 * (_phase(n, r0, z0, rng.random()) / w) ** 2)
        s -= s.mean()
        x += (s * (snr / s.norm())).float()
        for h in range(1, 9):
            if snr * snr * share[h - 1] >= 30.0 and abs(h * z0) <= zmax and h * r0 < n / 2 - 2048:
                truth.append((h * r0, h * z0))
    for _ in range(chirps):
        r0, z0 = rng.uniform(0.05, 0.9) * n / 2, rng.uniform(-0.9, 0.9) * zmax
        power = rng.uniform(40.0, 200.0)              # N a^2 / 2 at the cell's centre
        x += (math.sqrt(2.0 * power / n) * torch.cos(2.0 * math.pi * _phase(n, r0, z0, rng.random()))).float()
        truth.append((r0, z0))
    return x, truth


def _normalised_spectrum(x):
    X = torch.fft.rfft(x)[:-1]
    X[0] = 0
    s2 = X.abs().double().square().sum() / (X.numel() - 1)
    return X * torch.sqrt(2.0 / s2).to(X.real.dtype)


def _config(c, max_peaks):
    return fd.make_config(c["n"], c["zmax"], c["taps"], c["seg"], precision=c["prec"], max_harm=c.get("harm", 1),
                          thr=(30.0,) * 5 if c.get("low") else THR, max_peaks=max_peaks,
                          norm_block=c.get("norm_block", 0), harm_mode=c.get("harm_mode", 0))


def _records(peaks, npeaks):
    """The peak records as a program reads them: bin, row, level and series as integers, the powers."""
    words = peaks.view(torch.int32).view(-1, 4)
    return {"npeaks": npeaks, "where": words[:, :3], "power": peaks.view(torch.float32).view(-1, 4)[:, 3]}


def _batch_shapes(c):
    rng = random.Random(c["pick"])
    shapes = []
    for i in range(c["series"]):
        n = 1 << (c["log2_hi"] if i == 0 else rng.randint(c["log2_lo"], c["log2_hi"]))
        zmax = rng.choice([20, 50, 84])
        shapes.append((n, zmax, {20: 64, 50: 128, 84: 256}[zmax]))
    return shapes


def _points(truth, count, n, zmax, seed):
    """Seeds within half a bin (in r and in z) of the injected signals."""
    g = _gen(seed + 1)
    t = torch.tensor(truth, dtype=torch.float64, device=DEV)
    pick = torch.randint(0, t.shape[0], (count,), generator=g, device=DEV)
    off = torch.rand(count, 2, generator=g, device=DEV, dtype=torch.float64) - 0.5
    return (t[pick] + off).contiguous()


def _cand_inputs(c, seed):
    """A normalised spectrum with some fifty signals in it, and points near them."""
    count = c["cands"] if c["kind"] == "refine" else c["points"]
    x, truth = _series(c["n"], c["zmax"], seed, chirps=48, trains=2)
    X = _normalised_spectrum(x)
    return X, _points(truth, count, c["n"], c["zmax"], seed)


def _noise_plane(c, seed):
    """Exponential cells of mean 2 (the law of noise in the plane) with harmonic families on top."""
    K, nb = c["zmax"] + 1, c["n"] // 2
    p = torch.empty(K, nb, device=DEV).exponential_(0.5, generator=_gen(seed))
    rng = random.Random(int(seed))
    for _ in range(40):
        r0, z0 = rng.randrange(64, nb // 16), 2 * rng.randint(-c["zmax"] // 32, c["zmax"] // 32)
        for h in range(1, 17):
            if abs(h * z0) <= c["zmax"]:
                p[(h * z0 + c["zmax"]) // 2, h * r0] += rng.uniform(5.0, 40.0)
    return p.to(torch.bfloat16) if c["prec"] == "bf16" else p


# ------------------------------------------------------------------------------ the cases
def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "search":
        s = fd.Search(_config(c, 16384), device=DEV)
        x, _ = _series(c["n"], c["zmax"], seed)
        return dict(kind=kind, search=s, series=x, out=dict(_records(s.peaks, s.npeaks), plane=s.plane_2d()))
    if kind == "batch":
        shapes = _batch_shapes(c)
        b = BatchSearch([fd.make_config(n, z, m, 2048 if c["prec"] == "fp32" else 8192, precision=c["prec"], max_harm=16,
                                        thr=THR, max_peaks=4096) for n, z, m in shapes], device=DEV, lanes=c["lanes"])
        x = torch.cat([_series(n, z, seed * 1000 + i, trains=i % 3)[0] for i, (n, z, _) in enumerate(shapes)])
        return dict(kind=kind, batch=b, series=x, out=_records(b.peaks, b.npeaks))
    if kind == "spectrum":
        plan = fd.fdas_plan(fd.make_config(c["n"], 0, 32, 1024, norm_block=c.get("norm_block", 0)))
        fd.fdas_make_templates(plan)
        x, _ = _series(c["n"], 20, seed, trains=1)
        return dict(kind=kind, plan=plan, series=x,
                    ws=torch.empty(plan.info.workspace_bytes, dtype=torch.uint8, device=DEV),
                    xhat=torch.empty(c["n"], device=DEV), sigma2=torch.zeros(1, dtype=torch.float64, device=DEV))
    if kind == "plane":
        plan = fd.fdas_plan(_config(c, 0))
        fd.fdas_make_templates(plan)
        X = _normalised_spectrum(_series(c["n"], c["zmax"], seed)[0])
        return dict(kind=kind, plan=plan, xhat=torch.view_as_real(X).reshape(-1).contiguous(),
                    ws=torch.empty(plan.info.workspace_bytes, dtype=torch.uint8, device=DEV),
                    plane=torch.empty(plan.info.K, plan.info.nb, dtype=plan.plane_dtype(), device=DEV))
    if kind == "peaks":
        plan = fd.fdas_plan(fd.make_config(c["n"], c["zmax"], 32, 1024, precision=c["prec"], max_harm=c["harm"],
                                           thr=THR_LOW, max_peaks=1 << 16, harm_mode=c.get("harm_mode", 0)))
        fd.fdas_make_templates(plan)
        peaks = torch.zeros(16 << 16, dtype=torch.uint8, device=DEV)
        npeaks = torch.zeros(1, dtype=torch.int32, device=DEV)
        return dict(kind=kind, plan=plan, plane=_noise_plane(c, seed), peaks=peaks, npeaks=npeaks,
                    ws=torch.empty(plan.info.workspace_bytes, dtype=torch.uint8, device=DEV),
                    out=_records(peaks, npeaks))
    plan = fd.fdas_plan(fd.make_config(c["n"], 2, c["taps"], 2048))
    X, pts = _cand_inputs(c, seed)
    s = dict(kind=kind, plan=plan, xhat=torch.view_as_real(X).reshape(-1).contiguous())
    if kind == "refine":
        return dict(s, seeds=pts, steps=c["steps"])
    return dict(s, fp64=c["fp64"], r=pts[:, 0].clone().requires_grad_(), z=pts[:, 1].clone().requires_grad_(),
                weight=torch.rand(pts.shape[0], generator=_gen(seed + 2), device=DEV, dtype=torch.float64) + 0.5)


def run(state):
    s, kind = state, state["kind"]
    if kind == "search":
        s["search"].search(s["series"])
        return s["out"]
    if kind == "batch":
        s["batch"].search(s["series"])
        return s["out"]
    if kind == "spectrum":
        ft.fdas_spectrum(s["plan"], s["series"], s["ws"], s["xhat"], s["sigma2"])
        return {"xhat": s["xhat"], "sigma2": s["sigma2"]}
    if kind == "plane":
        ft.fdas_plane(s["plan"], s["xhat"], s["ws"], s["plane"])
        return s["plane"]
    if kind == "peaks":
        ft.fdas_peaks(s["plan"], s["plane"], s["ws"], s["peaks"], s["npeaks"])
        return s["out"]
    if kind == "refine":
        out, power, evals = rf.refine(s["plan"], s["xhat"], s["seeds"], s["steps"])
        return {"points": out, "power": power, "evals": evals}
    p = rf.interp_power(s["plan"], s["xhat"], s["r"], s["z"], fp64=s["fp64"])
    gr, gz = torch.autograd.grad(p, (s["r"], s["z"]), grad_outputs=s["weight"])
    return {"power": p.detach(), "dr": gr, "dz": gz}


# ------------------------------------------------------------------------------ necessary work
def _plane_flops(n, zmax, taps):
    """The overlap-save form at its cheapest power-of-two segment length: one segment FFT, then per
    template a complex product, an inverse FFT and the powers."""
    nb, K, best = n // 2, zmax + 1, None
    for lg in range(6, 15):
        S = 1 << lg
        if S < 2 * taps:
            continue
        L = S - taps + 1
        f = nb / L * (5.0 * S * lg + K * (6.0 * S + 5.0 * S * lg + 3.0 * L))
        best = f if best is None else min(best, f)
    return best


def _gathers(n, zmax, harm):
    g, H = 0, 2
    while H <= harm:
        g += (2 * (zmax // H // 2) + 1) * (n // 2 // H) * (H // 2)
        H *= 2
    return g


def work(case):
    c, kind = case, case["kind"]
    if kind in ("search", "plane"):
        eb = 2 if c["prec"] in ("bf16", "bf16_direct") else 4
        cells = (c["zmax"] + 1) * (c["n"] // 2)
        f = _plane_flops(c["n"], c["zmax"], c["taps"])
        if kind == "search":
            f += 2.5 * c["n"] * math.log2(c["n"]) + _gathers(c["n"], c["zmax"], c["harm"])
        return {"bytes": 4 * c["n"] + cells * eb, "flops": f}
    if kind == "batch":
        shapes = _batch_shapes(c)
        return {"bytes": sum(4 * n for n, _, _ in shapes),
                "flops": sum(_plane_flops(n, z, m) + 2.5 * n * math.log2(n) + _gathers(n, z, 16) for n, z, m in shapes)}
    if kind == "spectrum":
        return {"bytes": 8 * c["n"], "flops": 2.5 * c["n"] * math.log2(c["n"])}
    if kind == "peaks":
        return {"bytes": (c["zmax"] + 1) * (c["n"] // 2) * (2 if c["prec"] == "bf16" else 4),
                "flops": _gathers(c["n"], c["zmax"], c["harm"])}
    # per evaluation and tap: three complex multiply-adds with the response's moments
    if kind == "refine":
        return {"bytes": 4 * c["n"] + 60 * c["cands"], "flops": 24.0 * c["taps"] * c["cands"] * (c["steps"] + 3)}
    return {"bytes": 4 * c["n"] + 56 * c["points"], "flops": 24.0 * c["taps"] * c["points"]}


# ------------------------------------------------------------------------------ 64-bit values
def _gauss(cycles):
    """Gauss-Legendre nodes and weights on [0, 1]: panels of 16 points, at most two cycles each."""
    x, w = np.polynomial.legendre.leggauss(16)
    panels = int(math.ceil(cycles / 2.0)) + 2
    mid = (np.arange(panels) + 0.5)[:, None] / panels
    u = (mid + 0.5 / panels * x[None, :]).reshape(-1)
    return (torch.tensor(u, device=DEV), torch.tensor(np.tile(0.5 / panels * w, panels), device=DEV))


def _cis(cycles):
    c = cycles - torch.round(cycles)
    return torch.polar(torch.ones_like(c), 2.0 * math.pi * c)


def _bank(zmax, m):
    """Unit-norm responses T_z(q), [K][m] complex128."""
    u, w = _gauss(zmax + m)
    q = torch.arange(-(m // 2), m - m // 2, dtype=torch.float64, device=DEV)
    z = torch.arange(-zmax, zmax + 1, 2, dtype=torch.float64, device=DEV)
    T = (_cis(0.5 * z[:, None] * u * u) * w) @ _cis(-u[:, None] * q)
    return T / T.abs().square().sum(1, keepdim=True).sqrt()


def _spectrum64(x, norm_block):
    X = torch.fft.rfft(x.double())[:-1]
    X[0] = 0
    s2 = X.abs().square().sum() / (X.numel() - 1)
    if not norm_block:
        return X * torch.sqrt(2.0 / s2), s2
    p = X.abs().square()
    p[0] = math.inf
    p = p.view(-1, norm_block).sort(1).values
    rank = torch.full((p.shape[0],), (norm_block - 1) // 2, device=DEV)
    rank[0] = (norm_block - 2) // 2
    med = p.gather(1, rank[:, None])
    return (X.view(-1, norm_block) * torch.sqrt(2.0 * math.log(2.0) / med)).reshape(-1), s2


def _plane64(X, zmax, m):
    S, nb = 16384, X.numel()
    L = S - m + 1
    segs = -(-nb // L)
    xp = torch.zeros(segs * L + S, dtype=torch.complex128, device=DEV)
    xp[m // 2: m // 2 + nb] = X
    Y = torch.fft.fft(xp.as_strided((segs, S), (L, 1)))
    T = _bank(zmax, m)
    out = torch.empty(T.shape[0], nb, dtype=torch.float64, device=DEV)
    for i in range(T.shape[0]):
        out[i] = torch.fft.ifft(Y * torch.fft.fft(T[i], S).conj())[:, :L].reshape(-1)[:nb].abs().square()
    return out


def _peaks64(plane, zmax, harm, thr, cap):
    """The peak list's powers by the definition: S_H over the harmonics, threshold, 3x3 local maximum."""
    p, nb, powers, H, lvl = plane.double(), plane.shape[1], [], 1, 0
    while H <= harm:
        zl = 2 * (zmax // H // 2)
        z = torch.arange(-zl, zl + 1, 2, device=DEV)
        n = (nb - 1) // H + 1
        s = torch.zeros(z.numel(), n, dtype=torch.float64, device=DEV)
        for h in range(1, H + 1):
            s += p[(h * z + zmax) // 2][:, : h * (n - 1) + 1: h]
        t = torch.full((s.shape[0] + 2, n + 2), -math.inf, dtype=torch.float64, device=DEV)
        t[1:-1, 1:-1] = s
        ok = s > thr[lvl]
        for di in (-1, 0, 1):
            for dr in (-1, 0, 1):
                if di or dr:
                    o = t[1 + di: 1 + di + s.shape[0], 1 + dr: 1 + dr + n]
                    ok &= (s > o) if (di, dr) < (0, 0) else (s >= o)
        powers.append(s[ok])
        H, lvl = 2 * H, lvl + 1
    v = torch.cat(powers)[:cap]
    out = torch.zeros(cap, dtype=torch.float64, device=DEV)
    out[: v.numel()] = v
    return out


class _Interp64:
    """P, dP/dr, dP/dz in 64 bits: the integral over u of the window's transform, which does not
    depend on the point, times the chirp exp(-i pi z u^2) and the offset from the anchor."""

    def __init__(self, X, m, r, zspan):
        k0 = torch.floor(r + 0.5).long()
        j = torch.arange(-(m // 2), m - m // 2, device=DEV)
        k = k0[:, None] + j
        win = torch.where((k >= 0) & (k < X.numel()), X[k.clamp(0, X.numel() - 1)], 0).to(torch.complex128)
        self.k0 = k0.double()
        self.u, w = _gauss(m // 2 + zspan + 2)
        self.B = (win @ _cis(self.u * j.double()[:, None])) * w

    def __call__(self, r, z):
        u = self.u
        e = self.B * _cis(-0.5 * z[:, None] * u * u - (r - self.k0)[:, None] * u)
        A, Y1, Y2 = e.sum(1), (e * u).sum(1), (e * u * u).sum(1)
        dr = 2.0 * (A.conj() * (-2j * math.pi * Y1)).real
        dz = 2.0 * (A.conj() * (-1j * math.pi * Y2)).real
        return A.abs().square(), dr, dz


def _ascend64(f, r, z, steps):
    P, gr, gz = f(r, z)
    alive = torch.ones_like(P, dtype=torch.bool)
    for _ in range(steps):
        s = 1.0 / (2.0 * math.pi ** 2 * P)
        dr, dz = (48.0 * gr - 90.0 * gz) * s, (-90.0 * gr + 180.0 * gz) * s
        sc = torch.maximum(4.0 * dr.abs(), dz.abs()).clamp(min=1.0)
        dr, dz, done = dr / sc, dz / sc, ~alive
        for _ in range(4):
            if bool(done.all()):
                break
            P2, gr2, gz2 = f(r + dr, z + dz)
            take = ~done & (P2 >= P)
            r, z = torch.where(take, r + dr, r), torch.where(take, z + dz, z)
            P, gr, gz = torch.where(take, P2, P), torch.where(take, gr2, gr), torch.where(take, gz2, gz)
            done = done | take
            dr, dz = 0.5 * dr, 0.5 * dz
        alive = alive & done
        if not bool(alive.any()):
            break
    return r, z, P, gr, gz


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "batch":
        return None                      # peak lists only: integers, and sums over a plane that is not returned
    if kind == "search":
        x, _ = _series(c["n"], c["zmax"], seed)
        X, _ = _spectrum64(x, c.get("norm_block", 0))
        return {"npeaks": None, "where": None, "power": None, "plane": _plane64(X, c["zmax"], c["taps"])}
    if kind == "spectrum":
        X, s2 = _spectrum64(_series(c["n"], 20, seed, trains=1)[0], c.get("norm_block", 0))
        return {"xhat": torch.view_as_real(X).reshape(-1), "sigma2": s2.reshape(1)}
    if kind == "plane":
        X = _normalised_spectrum(_series(c["n"], c["zmax"], seed)[0])
        return _plane64(X.to(torch.complex128), c["zmax"], c["taps"])
    if kind == "peaks":
        if c["prec"] != "fp32" or c.get("harm_mode", 0):
            return None
        return {"npeaks": None, "where": None, "power": _peaks64(_noise_plane(c, seed), c["zmax"], c["harm"], THR_LOW, 1 << 16)}
    X, pts = _cand_inputs(c, seed)
    r, z = pts[:, 0].contiguous(), pts[:, 1].contiguous()
    f = _Interp64(X, c["taps"], r, c["zmax"] + 24)
    if kind == "refine":
        r, z, P, gr, gz = _ascend64(f, r, z, c["steps"] + 1)
        return {"points": torch.stack([r, z], 1), "power": torch.stack([P, gr, gz], 1), "evals": None}
    P, gr, gz = f(r, z)
    g = torch.rand(pts.shape[0], generator=_gen(seed + 2), device=DEV, dtype=torch.float64) + 0.5
    return {"power": P, "dr": g * gr, "dz": g * gz}
