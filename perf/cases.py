"""The workloads that this library's speed is measured on.

A case is one call a user of the library makes on a file that is already in GPU
memory: dedispersion, spectra, power planes, whole searches, the single-pulse
search and folding.  The sizes are those of the workloads in
``paper_1912_12807_gb300/synth.py`` (64-channel test file, 256-channel
drift-scan file, 96-channel 1-bit survey file, 200-channel file with the
six-row plan of the paper's Table 3), smaller and ragged relatives of them, and
files with masked channels and more than 256 of them.

Files are made on the GPU from the seed: Gaussian noise quantised to 8 bits (or
fair bits), a few faint dispersed pulsars, narrowband interference and a
broadband burst.  A program that searches a series of files keeps one context
and one plan for all files of a shape, and so does ``prepare``.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1912_12807_gb300 import pss, synth

K_DISP = 4.148808e3  # s MHz^2 pc^-1 cm^3

DRIFT = dict(nchan=256, nsamp=1 << 18, nbits=8, tsamp=2e-4, lo=1050.0, hi=1450.0, masked=0, rfi=3)
SMALL = dict(nchan=64, nsamp=1 << 16, nbits=8, tsamp=2e-4, lo=1200.0, hi=1500.0, masked=0, rfi=0)
SURVEY = dict(nchan=96, nsamp=1000003, nbits=1, tsamp=2.5e-4, lo=1230.0, hi=1518.0, masked=0, rfi=0)
FAST = dict(nchan=200, nsamp=1 << 18, nbits=8, tsamp=2e-4, lo=290.0, hi=340.0, masked=0, rfi=2)
SEARCH = dict(zmax=0, numharm=8)

# plan rows "dm_lo:dm_step:n_dm:ds"
SURVEY_PLAN = "0:0.5:400:1,200:1:400:2,600:5:281:4"
TABLE3_PLAN = "0:0.1:315:8,31.5:0.2:157:16,62.9:0.5:153:32,139.4:1:139:64,278.4:2:139:128,556.4:3:76:128"


def listed():
    return [
        # the smallest call: a short file and a few trials, e.g. around a known pulsar
        dict(SMALL, name="dedisperse_small", op="dedisperse", nsamp=1 << 14, plan="40:1:21:1"),
        # every trial of a drift-scan file, as prepsubband makes them for other programs
        dict(DRIFT, name="dedisperse_driftscan", op="dedisperse", plan="0:0.5:1001:1"),
        # a long 1-bit survey pointing of ragged length with a staged plan
        dict(SURVEY, name="dedisperse_survey_1bit", op="dedisperse", plan=SURVEY_PLAN),
        # whitened spectra of a ragged file with masked channels, more than 256 of them kept
        dict(DRIFT, **SEARCH, name="spectrum_masked", op="spectrum", nchan=400, nsamp=200003, masked=57, plan="0:1:128:1"),
        # power planes without acceleration
        dict(SMALL, **SEARCH, name="plane_small", op="plane", plan="0:1:101:1"),
        # f-fdot planes of a few trials of a drift-scan file
        dict(DRIFT, name="plane_accel", op="plane", plan="100:1:8:1", rfi=0, zmax=200, numharm=8),
        # whole searches: the test file, the drift-scan file, the same with acceleration, the six-row plan
        dict(SMALL, **SEARCH, name="search_small", op="search", plan="0:1:101:1"),
        dict(DRIFT, name="search_driftscan", op="search", plan="0:0.5:1001:1", zmax=0, numharm=16),
        dict(DRIFT, name="search_accel", op="search", plan="0:1:301:1", rfi=0, zmax=200, numharm=8),
        dict(FAST, name="search_table3", op="search", plan=TABLE3_PLAN, zmax=0, numharm=16),
        # boxcar events of every trial of a drift-scan file
        dict(DRIFT, name="single_pulse_driftscan", op="single_pulse", plan="0:0.5:1001:1"),
        # the best candidates of a drift-scan file folded
        dict(DRIFT, name="fold_driftscan", op="fold", plan="0:0.5:1001:1", ncand=64, nbin=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    """One more case: any operation on a file between the smallest and the drift-scan or survey
    file, of any length (odd ones included), with a one-row or a staged plan."""
    op = rng.choice(["dedisperse", "dedisperse", "spectrum", "plane", "search", "search", "single_pulse", "fold"])
    kind = rng.choice(["small", "drift", "drift", "survey", "fast"])
    base = {"small": SMALL, "drift": DRIFT, "survey": SURVEY, "fast": FAST}[kind]
    c = dict(base, op=op)
    if kind == "survey":
        c["nchan"] = 8 * rng.randint(4, 16)
        c["nsamp"] = _log(rng, 1 << 16, 1 << 20) | 1
        n = _log(rng, 8, 200)
        c["plan"] = "0:0.5:%d:1,%g:1:%d:2,%g:5:%d:4" % (n, 0.5 * n, max(1, n // 2), 0.5 * n + max(1, n // 2), max(1, n // 3))
    elif kind == "fast":
        c["nchan"] = rng.randint(100, 300)
        c["nsamp"] = _log(rng, 1 << 17, 1 << 18)
        n, ds = _log(rng, 20, 300), rng.choice([8, 16, 32])
        c["plan"] = "0:0.1:%d:%d,%g:0.3:%d:%d" % (n, ds, 0.1 * n, max(1, n // 2), 2 * ds)
    else:
        c["nchan"] = _log(rng, 32, 96) if kind == "small" else _log(rng, 128, 600)
        c["nsamp"] = _log(rng, 1 << 14, 1 << 17) if kind == "small" else _log(rng, 1 << 16, 1 << 18)
        c["masked"] = rng.choice([0, 0, c["nchan"] // rng.randint(6, 20)])
        most = 512 if c["nchan"] <= 256 else 256
        c["plan"] = "%g:%g:%d:%d" % (rng.choice([0, 25, 60]), rng.choice([0.25, 0.5, 1.0]), _log(rng, 8, most), rng.choice([1, 1, 1, 2]))
    if op in ("spectrum", "plane", "search"):
        c["zmax"] = 0 if op == "spectrum" else rng.choice([0, 0, 20, 50, 100, 200])
        c["numharm"] = rng.choice([8, 16]) if op == "search" else 8
        # planes are large: at most the work of the largest listed acceleration search / plane
        if c["zmax"]:
            most = 128 if op == "search" else 6
            rows = [r.split(":") for r in c["plan"].split(",")]
            c["rfi"] = 0  # a file searched for acceleration has its interference removed
            c["plan"] = ",".join("%s:%s:%d:%s" % (r[0], r[1], min(int(r[2]), most), r[3]) for r in rows[:1])
    if op == "fold":
        c["ncand"], c["nbin"] = _log(rng, 4, 128), rng.choice([32, 64, 100, 128])
    return c


# ---------------------------------------------------------------------------
# files
# ---------------------------------------------------------------------------

def _freqs(case):
    foff = (case["hi"] - case["lo"]) / case["nchan"]
    return case["lo"] + 0.5 * foff + foff * np.arange(case["nchan"])


def _rows(case):
    return [tuple(float(v) for v in r.split(":")) for r in case["plan"].split(",")]


def _mask(case):
    """Kept channels: `masked` of them (fixed by the case) removed, None where all are kept."""
    if not case["masked"]:
        return None
    m = np.ones(case["nchan"], dtype=np.uint8)
    m[np.random.RandomState(case["nchan"]).permutation(case["nchan"])[: case["masked"]]] = 0
    return m


def _pulsars(case, seed):
    """A few faint sources inside the plan's DM range: (period, DM, duty, phase, folded S/N)."""
    r = np.random.RandomState(seed % (1 << 31))
    rows = _rows(case)
    dm_hi = rows[-1][0] + rows[-1][1] * rows[-1][2]
    ds = rows[0][3]
    out = []
    for _ in range(4):
        period = math.exp(r.uniform(math.log(max(0.005, 8 * ds * case["tsamp"])), math.log(0.5)))
        out.append((period, r.uniform(rows[0][0], dm_hi), r.uniform(0.03, 0.1), r.uniform(), r.uniform(25.0, 60.0)))
    return out


def _make_file(case, seed):
    """File bytes on the GPU: uint8 [nsamp][nchan], or [nsamp][nchan / 8] most significant bit first."""
    nchan, nsamp, ts = case["nchan"], case["nsamp"], case["tsamp"]
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    f = torch.from_numpy(_freqs(case)).to(dev)
    dly = K_DISP * (1.0 / (f * f) - 1.0 / (f.max() * f.max()))  # per unit DM
    psrs = _pulsars(case, seed)
    r = np.random.RandomState((seed + 1) % (1 << 31))
    rfi = [int(c) for c in r.permutation(nchan)[: case["rfi"]]]
    burst = int(0.37 * nsamp)
    chunks = []
    step = max(1, (1 << 24) // nchan)
    for s0 in range(0, nsamp, step):
        n = min(step, nsamp - s0)
        t = (s0 + torch.arange(n, device=dev, dtype=torch.float64)) * ts
        x = torch.zeros((n, nchan), device=dev)
        for period, dm, duty, ph0, snr in psrs:
            ph = (t[:, None] - dm * dly[None, :]).mul_(1.0 / period).add_(ph0)
            d = (ph - torch.floor(ph + 0.5)).float()
            sig = duty / (2.0 * math.sqrt(2.0 * math.log(2.0)))
            x += snr / math.sqrt(nchan * nsamp * duty) * torch.exp(-0.5 * (d / sig) ** 2)
        lo, hi = max(0, burst - s0), min(n, burst + 25 - s0)
        if lo < hi and case.get("zmax", 0) == 0:
            x[lo:hi] += 4.0 if case["nbits"] == 8 else 0.6
        if case["nbits"] == 8:
            x += torch.randn((n, nchan), generator=g, device=dev)
            if rfi:
                x[:, rfi] += 3.0 * torch.sin(2.0 * math.pi * 50.0 * t)[:, None].float()
            chunks.append(torch.clamp(torch.round(128.0 + 16.0 * x), 0, 255).to(torch.uint8))
        else:
            bits = (torch.rand((n, nchan), generator=g, device=dev) < 0.5 + 0.4 * x).to(torch.uint8)
            w = torch.tensor([128, 64, 32, 16, 8, 4, 2, 1], device=dev, dtype=torch.uint8)
            chunks.append((bits.view(n, nchan // 8, 8) * w).sum(dim=2, dtype=torch.uint8))
    return torch.cat(chunks).contiguous()


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

_kept = {"key": None, "ctx": None, "plan": None}  # the handles of the shape at hand


def _handles(case):
    key = tuple(case[k] for k in ("op", "nchan", "nsamp", "nbits", "tsamp", "lo", "hi", "masked", "plan"))
    if _kept["key"] != key:
        f = _freqs(case)
        desc = pss.FilDesc(case["nchan"], case["nsamp"], case["tsamp"], float(f[0]), float(f[1] - f[0]), case["nbits"],
                           chan_mask=_mask(case))
        rows = [synth.Stage(a, b, int(n), int(ds)) for a, b, n, ds in _rows(case)]
        _kept.update(key=key, ctx=pss.Context(0), plan=pss.Plan(desc, rows))
    return _kept["ctx"], _kept["plan"]


def prepare(case, seed):
    """The file in GPU memory, the context and plan kept for its shape, and the search parameters;
    for folding also the list of candidates."""
    ctx, plan = _handles(case)
    s = {"op": case["op"], "ctx": ctx, "plan": plan, "data": _make_file(case, seed)}
    if "zmax" in case:
        s["cfg"] = pss.search_cfg(zmax=case["zmax"], numharm=case["numharm"])
    if case["op"] == "fold":
        # sifted candidates cluster around the sources' DMs, with their harmonics
        r = np.random.RandomState(seed % (1 << 31))
        dms = plan.dms()
        dm, fhz = [], []
        for k in range(case["ncand"]):
            period, d, _, _, _ = _pulsars(case, seed)[k % 4]
            near = int(np.argmin(np.abs(dms - d))) + int(r.randint(-2, 3))
            dm.append(min(max(near, 0), plan.ndm - 1))
            fhz.append((1 + k // 8 % 4) / period)
        s.update(dm_idx=np.array(dm), f_hz=np.array(fhz), fdot=r.uniform(-1e-3, 1e-3, case["ncand"]), nbin=case["nbin"])
    return s


def _buffer(found):
    """The whole buffer that a call filled with the candidates it found (zero after the last one):
    its length does not depend on how many there are."""
    return found if found.base is None else found.base


def run(s):
    op, ctx, plan, data = s["op"], s["ctx"], s["plan"], s["data"]
    if op == "dedisperse":
        return pss.pss_dedisperse(ctx, plan, data, 0, plan.ndm)
    if op == "spectrum":
        return pss.pss_spectrum(ctx, plan, data, s["cfg"], 0, plan.ndm)
    if op == "plane":
        return pss.pss_power_plane(ctx, plan, data, s["cfg"], 0, plan.ndm)
    if op == "search":
        c = _buffer(pss.pss_search_dm_batch(ctx, plan, data, s["cfg"], 0, plan.ndm))
        out = {k: c[k] for k in ("dm_idx", "numharm", "dm", "r", "z", "f_hz", "power", "dm_hits", "h", "j")}
        out["sigma"] = c["sigma"].astype(np.float32)  # a function of the 32-bit power
        return out
    if op == "single_pulse":
        e = _buffer(pss.pss_single_pulse(ctx, plan, data, 0, plan.ndm))
        return {k: e[k] for k in ("dm_idx", "width", "t", "boxsum", "snr")}
    prof, cnt, res = pss.pss_fold(ctx, plan, data, s["dm_idx"], s["f_hz"], s["fdot"], nbin=s["nbin"], nfreq=9, step_bins=0.25)
    return {"profiles": prof, "counts": cnt, "f_hz": res["f_hz"], "chi2_red": res["chi2_red"], "best": res["best"]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _shape(case):
    """Per plan row: (trials, samples per trial, transform length), with the library's rules
    (one valid length per file, the next power of two), and the kept channels."""
    m = _mask(case)
    f = _freqs(case)
    f_ref = f.max()
    rows = _rows(case)
    d_max = 0
    for lo, step, n, _ in rows:
        v = K_DISP * (lo + (n - 1) * step) * (1.0 / (f * f) - 1.0 / (f_ref * f_ref)) / case["tsamp"]
        d_max = max(d_max, int(np.floor(v.max() + 0.5)))
    out = []
    for _, _, n, ds in rows:
        nv = (case["nsamp"] - d_max) // int(ds)
        out.append((int(n), nv, 1 << (nv - 1).bit_length()))
    return out, case["nchan"] if m is None else int(m.sum())


def work(case):
    """The file read once, and the outputs written once; one addition per kept channel, output
    sample and native sample, 5 N log2 N / 2 per real transform, and the plane, harmonic and
    boxcar arithmetic."""
    rows, ck = _shape(case)
    ds = [int(r[3]) for r in _rows(case)]
    nbytes = case["nsamp"] * case["nchan"] * case["nbits"] // 8
    op = case["op"]
    if op == "fold":
        used = min(sum(n for n, _, _ in rows), case["ncand"], 20)  # distinct trials near four sources
        nv = max(nv for _, nv, _ in rows)
        return {"bytes": nbytes + 16.0 * case["ncand"] * case["nbin"], "flops": float(used * nv * ck + 3 * 9 * case["ncand"] * nv)}
    flops = float(sum(n * nv * d * ck for (n, nv, _), d in zip(rows, ds)))
    if op == "dedisperse":
        return {"bytes": float(nbytes + sum(4 * n * nv for n, nv, _ in rows)), "flops": flops}
    if op == "single_pulse":
        return {"bytes": float(nbytes), "flops": flops + sum(2.0 * len(pss.SP_WIDTHS) * n * nv for n, nv, _ in rows)}
    flops += sum(n * 2.5 * nf * math.log2(nf) for n, _, nf in rows)
    if op == "spectrum":
        return {"bytes": float(nbytes + sum(4 * n * nf for n, _, nf in rows)), "flops": flops}
    nz = case["zmax"] + 1 if case["zmax"] else 1  # steps of 2 in z
    per = 70.0 if case["zmax"] else 64.0  # overlap-save correlation, or the 32 real taps of every second value
    flops += sum(per * n * nz * nf for n, _, nf in rows)
    if op == "plane":
        return {"bytes": float(nbytes + sum(4 * n * nz * nf for n, _, nf in rows)), "flops": flops}
    return {"bytes": float(nbytes), "flops": flops + sum(float(case["numharm"]) * n * nz * nf for n, _, nf in rows)}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------

def _exact_taps(z, parity, m):
    """conj(rho(parity/2 - t, z)), t = -m+1 .. m, by composite Gauss-Legendre quadrature of
    rho(q, z) = int_0^1 exp(2 pi i ((q - z/2) u + z u^2 / 2)) du."""
    x, w = np.polynomial.legendre.leggauss(16)
    panels = 160
    u = ((np.arange(panels)[:, None] + 0.5 * (x[None, :] + 1.0)) / panels).reshape(-1)
    wt = np.tile(0.5 * w / panels, panels)
    u, wt = torch.from_numpy(u).cuda(), torch.from_numpy(wt).cuda()
    q = 0.5 * parity - torch.arange(-m + 1, m + 1, device="cuda", dtype=torch.float64)
    ph = (q[:, None] - 0.5 * z) * u[None, :] + 0.5 * z * (u * u)[None, :]
    ph = 2.0 * math.pi * (ph - torch.floor(ph))
    return torch.complex((torch.cos(ph) * wt).sum(1), -(torch.sin(ph) * wt).sum(1))


def _exact_spectra(case, seed):
    """Whitened half spectra, one [nfft/2] complex128 tensor per trial."""
    data = _make_file(case, seed)
    if case["nbits"] == 1:
        shift = torch.arange(7, -1, -1, device="cuda", dtype=torch.uint8)
        data = ((data[:, :, None] >> shift) & 1).view(case["nsamp"], case["nchan"])
    x = data.t().contiguous()
    m = _mask(case)
    f = _freqs(case)
    f_ref = f.max()
    keep = np.arange(case["nchan"]) if m is None else np.nonzero(m)[0]
    shapes, _ = _shape(case)
    inv = 1.0 / (f * f) - 1.0 / (f_ref * f_ref)
    for (lo, step, n, ds), (_, nv, nfft) in zip(_rows(case), shapes):
        ds = int(ds)
        for i in range(int(n)):
            d = np.floor(((K_DISP * (lo + i * step)) * inv) / case["tsamp"] + 0.5).astype(np.int64)
            s = torch.zeros(nv * ds, device="cuda", dtype=torch.int32)
            for c in keep:
                s += x[c, d[c]:d[c] + nv * ds]
            y = s.view(nv, ds).sum(1).double()
            y = torch.nn.functional.pad(y - y.mean(), (0, nfft - nv))
            a = torch.fft.rfft(y)[: nfft // 2]
            a[0] = 0
            p = (a.abs() ** 2).view(-1, 1024).sort(dim=1).values
            med = p[:, 511].clone()
            med[0] = p[0, 1:][511]  # the DC bin (0, sorted first) does not count: 1023 values, rank 511
            g = torch.where(med > 0, math.log(2.0) / med, torch.zeros_like(med)).sqrt()
            yield (a.view(-1, 1024) * g[:, None]).view(-1)


def exact(case, seed):
    """Spectra and planes in 64 bits; the other operations return integers, or values decided by
    comparisons of 32-bit sums."""
    if case["op"] not in ("spectrum", "plane"):
        return None
    if sum(n * case["nchan"] for n, _, _ in _shape(case)[0]) > 120000:
        return None
    spectra = _exact_spectra(case, seed)
    if case["op"] == "spectrum":
        return torch.cat(list(spectra))
    zmax = case["zmax"]
    zs = [-zmax + 2.0 * j for j in range(zmax + 1)] if zmax else [0.0]
    rows = _shape(case)[0]
    if sum(n * nf for n, _, nf in rows) * len(zs) > 5.2e8:
        return None
    out = []
    taps = {}
    for a in spectra:
        M = a.numel()
        L = 2 * M if M > 4096 else 4 * M
        fa = torch.fft.fft(a, n=L)
        plane = torch.empty((len(zs), M, 2), device="cuda", dtype=torch.float64)
        for j, z in enumerate(zs):
            half = int(math.ceil(abs(z) / 2.0)) + 16
            for par in (0, 1):
                if (j, par) not in taps:
                    g = _exact_taps(z, par, half)
                    taps[j, par] = g / g.abs().square().sum().sqrt()
                # sum_t a[k + t] g[t], t = -half+1 .. half
                h = torch.zeros(L, device="cuda", dtype=torch.complex128)
                t = torch.arange(-half + 1, half + 1, device="cuda")
                h[(-t) % L] = taps[j, par]
                plane[j, :, par] = torch.fft.ifft(fa * torch.fft.fft(h))[:M].abs() ** 2
        out.append(plane.reshape(-1))
    return torch.cat(out)
