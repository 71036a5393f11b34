"""The work that a user of this package has it do, as measurable cases through its public calls.

A case is one call (or one forward and backward call) of `paper_1801_02391_gb300.frbx`: a whole search of one
scan, a fit of listed segments, a refinement step, a calibration, or a batched search of several scans.  The
setups are the ones of this repository's own workloads: the S-band layout (8 subbands x 32 points), the two
lower VGOS bands (16 x 64) and all four VGOS bands (32 x 64).  Inputs are noise with dispersed pulses and RFI
on flagged points, made on the GPU from the seed.
"""
import math

import numpy as np
import torch

from paper_1801_02391_gb300 import frbx

K_DM = 4.148808e6  # ms MHz^2 per (pc cm^-3), the physical constant, for injected pulses only

# setup: subband edges (MHz), points per subband, AP length (ms), share of flagged points, window lengths (APs)
SETUPS = {
    "sband": ([1400.0 + 32.0 * i for i in range(8)], 32, 1.0, 0.01, "2,4,8,16"),
    "two_band": ([b + 32.0 * i for b in (3000.0, 5464.0) for i in range(8)], 64, 1.0, 0.05, "2,4,8,16"),
    "vgos": ([b + 32.0 * i for b in (3000.0, 5464.0, 7960.0, 10424.0) for i in range(8)], 64, 0.5, 0.05, "1,2,4,8,16,32"),
}
BW = 32.0


def _search(name, setup, n_bl, n_dm, dm_hi, t, windows="", kernel=0, sbd_ns=0.0, host=False):
    return {"name": name, "do": "search", "setup": setup, "n_bl": n_bl, "n_dm": n_dm, "dm_hi": dm_hi, "t": t,
            "windows": windows or SETUPS[setup][4], "kernel": kernel, "sbd_ns": sbd_ns, "host": host}


def listed():
    return [
        # the S-band search at its configured size: 3 baselines, 101 DM trials, 4096 APs
        _search("search_sband", "sband", 3, 101, 1000.0, 4096),
        # a slice of the headline search: 20000-AP scans of the four-band setup, 3 of 15 baselines, 64 of 512 DMs
        _search("search_vgos", "vgos", 3, 64, 2000.0, 20000),
        # a short, ragged scan that arrives in pinned host memory
        _search("search_vgos_short_host", "vgos", 2, 16, 300.0, 2411, host=True),
        # the source position is known: a search window of +-64 ns around zero single-band delay
        _search("search_vgos_window", "vgos", 3, 32, 1500.0, 9973, sbd_ns=64.0),
        # the lower-precision form: one BF16 product per AP
        _search("search_vgos_bf16", "vgos", 2, 24, 600.0, 7000, kernel=7),
        # window lengths matched to expected pulse widths, no powers of two: every segment is fitted by itself
        _search("search_widths", "vgos", 1, 8, 200.0, 1501, windows="3,6,10"),
        # candidate follow-up: a few dozen segments looked at again
        {"name": "fit_few", "do": "fit", "setup": "vgos", "n_bl": 3, "n_dm": 40, "dm_hi": 800.0, "t": 3000, "n_seg": 40},
        # a long list of segments, as from another search's crossings
        {"name": "fit_many", "do": "fit", "setup": "vgos", "n_bl": 15, "n_dm": 64, "dm_hi": 1000.0, "t": 5003, "n_seg": 20000},
        # one candidate in a gradient-ascent loop: forward and backward
        {"name": "refine_one", "do": "refine", "setup": "sband", "n_bl": 3, "t": 1200, "n_cand": 1},
        # all candidates of a search refined at once
        {"name": "refine_many", "do": "refine", "setup": "vgos", "n_bl": 15, "t": 6000, "n_cand": 200},
        # channel delays and phases of 15 baselines from half a second of a calibrator
        {"name": "calibrate", "do": "calibrate", "setup": "vgos", "n_bl": 15, "t": 1200, "l": 1000},
        # scans of uneven length on all three setups in one call, with their series
        {"name": "batch", "do": "batch", "n_scans": 5, "n_bl": 4, "n_dm": 32, "dm_hi": 600.0, "t": 3300},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["search", "search", "search", "search", "fit", "refine", "calibrate", "batch"])
    setup = rng.choice(["sband", "two_band", "vgos", "vgos"])
    n_bl = rng.randint(1, 15)
    if do == "search":
        c = _search("", setup, n_bl, _log(rng, 2, 128), rng.choice([100.0, 300.0, 1000.0, 1500.0]), _log(rng, 300, 20000))
        del c["name"]
        form = rng.choice(["whole", "whole", "window", "host", "bf16", "e4m3", "fp32", "widths"])
        limit = {"sband": 6e6, "two_band": 4e6, "vgos": 2.5e6}[setup]
        if form == "window":
            c["sbd_ns"] = rng.choice([64.0, 200.0, 450.0])
        elif form == "host":
            c["host"] = True
        elif form in ("bf16", "e4m3") and setup != "sband":
            c["kernel"] = 7 if form == "bf16" else 8
        elif form == "fp32":
            c["kernel"], limit = 4, limit / 3
        elif form == "widths":
            c["windows"], limit = rng.choice(["3,6,10", "5,12", "1,3,9"]), limit / 40
        while c["n_bl"] * c["n_dm"] * c["t"] > limit:
            k = rng.choice(["n_bl", "n_dm", "t"])
            c[k] = max({"n_bl": 1, "n_dm": 2, "t": 300}[k], int(c[k] * 0.7))
        return c
    if do == "fit":
        return {"do": "fit", "setup": setup, "n_bl": n_bl, "n_dm": _log(rng, 2, 64), "dm_hi": 300.0, "t": _log(rng, 900, 5000),
                "n_seg": _log(rng, 1, 20000)}
    if do == "refine":
        return {"do": "refine", "setup": setup, "n_bl": n_bl, "t": _log(rng, 900, 6000), "n_cand": _log(rng, 1, 200)}
    if do == "calibrate":
        t = _log(rng, 60, 1500)
        return {"do": "calibrate", "setup": setup, "n_bl": n_bl, "t": t, "l": rng.randint(t // 2, t)}
    return {"do": "batch", "n_scans": rng.randint(2, 5), "n_bl": rng.randint(1, 4), "n_dm": _log(rng, 4, 32), "dm_hi": 600.0,
            "t": _log(rng, 800, 3300)}


# ---------------------------------------------------------------------------- inputs
class _Setup:
    """Frequencies, flags and grid sizes of a setup (the flags belong to the setup, not to the data)."""

    def __init__(self, name):
        f0, self.J, self.t_ap, share, _ = SETUPS[name]
        self.f0 = np.array(f0)
        self.N, self.C = len(f0), len(f0) * self.J
        self.f = (self.f0[:, None] + np.arange(self.J)[None, :] * BW / self.J).reshape(-1)
        self.flags = (np.random.RandomState(7).random_sample(self.C) < share).astype(np.uint8)
        self.used = (self.flags == 0) & (np.arange(self.C) % self.J > 0)
        self.g = np.rint((self.f0 - self.f0.min()) / BW).astype(np.int64)
        self.Ls, self.Lm = 2 * self.J, 2 * (1 << int(self.g.max()).bit_length())

    def handle(self):
        return frbx.Handle(self.f0, self.J, BW, self.t_ap, flag=self.flags)

    def shifts(self, dms):
        x = 0.5 + (4.15e6 * dms)[:, None] * (1.0 / (self.f * self.f) - 1.0 / (self.f.max() * self.f.max()))[None, :] / self.t_ap
        return np.floor(x).astype(np.int64)


def _cube(su, n_bl, t, dm_hi, gen, pulses=2):
    """Noise, RFI on the flagged points and dispersed pulses: complex64 [n_bl][t][C] on the GPU."""
    dev = "cuda"
    vis = torch.empty((n_bl, t, su.C), dtype=torch.complex64, device=dev)
    torch.view_as_real(vis).normal_(0.0, math.sqrt(0.5), generator=gen)
    scale = torch.from_numpy(np.where(su.flags, math.sqrt(31.0), 1.0).astype(np.float32)).to(dev)
    vis *= scale
    u = torch.rand((pulses, 4), generator=gen, device=dev, dtype=torch.float64).cpu().numpy()
    tau = torch.rand((n_bl, 2), generator=gen, device=dev, dtype=torch.float64) * 49.0 + 1.0
    f = torch.from_numpy(su.f).to(dev)
    for dm_u, t_u, w_u, s_u in u:
        delay = K_DM * dm_u * dm_hi * (su.f ** -2 - su.f.max() ** -2) / su.t_ap
        width = 1 + int(w_u * 9.99)
        a = (12.0 + 20.0 * s_u) / math.sqrt(width * int(su.used.sum()))
        k = torch.from_numpy(int(t_u * 0.7 * t) + np.rint(delay).astype(np.int64)).to(dev)
        sig = a * torch.exp(2j * math.pi * ((f - f[0])[None, :] * tau[:, :1] * 1e-3 + tau[:, 1:]))
        col = torch.arange(su.C, device=dev)
        for i in range(width):
            on = ((k + i) < t).to(torch.float64)
            vis[:, (k + i).clamp(max=t - 1), col] += (sig * on).to(torch.complex64)
    return vis


def _gen(seed, k=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1801_02391 + 1000 * int(seed) + k)
    return g


def _windows(case):
    return np.array([int(w) for w in case["windows"].split(",")], np.int32)


def _batch_scans(case):
    names = ["vgos", "sband", "two_band"]
    share = [1.0, 0.61, 0.83, 0.37, 0.52]
    return [(names[i % 3], max(300, int(case["t"] * share[i]) | 1)) for i in range(case["n_scans"])]


def _rows(case, su, gen, dms):
    n = case["n_seg"]
    u = torch.rand((n, 4), generator=gen, device="cuda", dtype=torch.float64).cpu().numpy()
    rows = np.zeros((n, 4), np.int32)
    rows[:, 0] = u[:, 0] * case["n_bl"]
    rows[:, 1] = u[:, 1] * len(dms)
    rows[:, 2] = np.array([1, 2, 4, 8, 16, 32])[(u[:, 2] * 6).astype(int)]
    rows[:, 3] = u[:, 3] * (case["t"] - su.shifts(dms).max(1)[rows[:, 1]] - rows[:, 2] + 1)
    return rows


def prepare(case, seed):
    do = case["do"]
    if do == "batch":
        handles, scans = {}, []
        for i, (name, t) in enumerate(_batch_scans(case)):
            su = _Setup(name)
            if name not in handles:
                handles[name] = su.handle()
            scans.append((handles[name], _cube(su, case["n_bl"], t, case["dm_hi"], _gen(seed, i), pulses=1)))
        return {"do": do, "batch": frbx.Batch(), "scans": scans, "dms": np.linspace(0.0, case["dm_hi"], case["n_dm"]),
                "windows": np.array([2, 4, 8, 16], np.int32)}
    su, gen = _Setup(case["setup"]), _gen(seed)
    s = {"do": do, "h": su.handle()}
    n_bl, t = case["n_bl"], case["t"]
    if do == "search":
        dms, win = np.linspace(0.0, case["dm_hi"], case["n_dm"]), _windows(case)
        vis = _cube(su, n_bl, t, case["dm_hi"], gen)
        n = n_bl * len(dms) * frbx.frbx_series_layout(t, win)[1]
        s.update(vis=vis.cpu().pin_memory() if case["host"] else vis, dms=dms, windows=win, kernel=case["kernel"],
                 combos=[(1 << n_bl) - 1] + ([0b011, 0b101] if n_bl == 3 else []),
                 sbd=(-case["sbd_ns"], case["sbd_ns"]) if case["sbd_ns"] else None,
                 series=torch.empty((n, 2), dtype=torch.int32, device="cuda"),
                 pnorm=torch.empty(n, dtype=torch.float32, device="cuda"))
    elif do == "fit":
        dms = np.linspace(0.0, case["dm_hi"], case["n_dm"])
        s.update(vis=_cube(su, n_bl, t, case["dm_hi"], gen), dms=dms, rows=_rows(case, su, gen, dms))
    elif do == "refine":
        s.update(_candidates(case, su, gen), vis=_cube(su, n_bl, t, 100.0, gen), fn=frbx.coherent_power_fn())
    else:
        s.update(vis=_calibrator(su, n_bl, t, gen), k0=(t - case["l"]) // 2, l=case["l"])
    return s


def _candidates(case, su, gen):
    n, n_bl = case["n_cand"], case["n_bl"]
    u = torch.rand((n, 2 + 3 * n_bl), generator=gen, device="cuda", dtype=torch.float64)
    p = torch.empty_like(u)
    dm_hi = min(600.0, 0.4 * case["t"] * su.t_ap / (K_DM * (su.f.min() ** -2 - su.f.max() ** -2)))
    p[:, 0] = u[:, 0] * dm_hi
    p[:, 1] = 10.0 + u[:, 1] * 0.4 * case["t"]
    p[:, 2::3] = u[:, 2::3] * 120.0 - 60.0
    p[:, 3::3] = u[:, 3::3] * 30.0 - 15.0
    p[:, 4::3] = u[:, 4::3] * 2.0 - 1.0
    width = torch.tensor([1, 2, 4, 8, 16], dtype=torch.int32, device="cuda")
    i = torch.randint(0, 5, (n,), generator=gen, device="cuda")
    return {"params": p.requires_grad_(True), "width": width[i].contiguous(),
            "dpower": torch.rand(n, generator=gen, device="cuda") + 0.5}


def _calibrator(su, n_bl, t, gen):
    """A strong continuous source: per baseline a delay, per channel a small delay and a phase of its own."""
    vis = _cube(su, n_bl, t, 100.0, gen, pulses=0)
    u = torch.rand((n_bl, 1 + 2 * su.N), generator=gen, device="cuda", dtype=torch.float64)
    f = torch.from_numpy(su.f).to("cuda")
    fj = torch.arange(su.C, device="cuda", dtype=torch.float64) % su.J * BW / su.J
    n = torch.arange(su.C, device="cuda") // su.J
    ph = ((f - f[0])[None, :] * (u[:, :1] * 40.0 - 20.0) * 1e-3 + (fj - BW / 2) * (u[:, 1 + n] - 0.5) * 4e-3 + u[:, 1 + su.N + n])
    vis += (0.4 * torch.exp(2j * math.pi * ph)).to(torch.complex64)[:, None, :]
    return vis


# ---------------------------------------------------------------------------- one pass
CAP = 4096  # candidate lists come back in arrays of this many rows, the rest zero


def _cands(a):
    """The candidates' numbers by type: series, DM, window, width, start, cells, windows, group | |G|, P | time, delays, DM."""
    n = min(len(a), CAP)
    whole, single, double = np.zeros((CAP, 9), np.int32), np.zeros((CAP, 2), np.float32), np.zeros((CAP, 4))
    whole[:n] = a.view(np.int32).reshape(-1, 20)[:n, :9]
    single[:n] = a.view(np.float32).reshape(-1, 20)[:n, 9:11]
    double[:n] = a.view(np.float64).reshape(-1, 10)[:n, 6:]
    return {"n": len(a), "whole": whole, "single": single, "double": double}


def _groups(a):
    n = min(len(a), CAP)
    whole = np.zeros((CAP, 3), np.int64)
    for i, k in enumerate(("bl_mask", "n_baselines", "n_pulses")):
        whole[:n, i] = a[k][:n]
    return {"n": len(a), "whole": whole}


def _segs(a):
    return {"amp": a["amp"], "sbd": a["sbd_idx"].view(np.int16), "mbd": a["mbd_idx"].view(np.int16)}


def run(s):
    do = s["do"]
    if do == "search":
        out = s["h"].search(s["vis"], s["dms"], s["windows"], combos=s["combos"], sbd_win_ns=s["sbd"], kernel=s["kernel"],
                            series_out=s["series"], pnorm_out=s["pnorm"])
        idx = s["series"].view(torch.int16)
        return {"amp": s["series"].view(torch.float32)[:, 0], "sbd": idx[:, 2], "mbd": idx[:, 3], "pnorm": s["pnorm"],
                "pulses": _cands(out["pulses"]), "combined": _cands(out["combined"]), "groups": _groups(out["groups"])}
    if do == "fit":
        return _segs(s["h"].fit_segments(s["vis"], s["dms"], s["rows"]))
    if do == "refine":
        power = s["fn"].apply(s["params"], s["h"], s["vis"], s["width"])
        grad, = torch.autograd.grad(power, s["params"], s["dpower"])
        return {"power": power, "grad": grad}
    if do == "calibrate":
        return dict(zip(("sbd", "mbd", "delay", "phase"), s["h"].calibrate(s["vis"], s["k0"], s["l"])))
    outs = s["batch"].search(s["scans"], s["dms"], s["windows"], want_series=True)
    return [{**_segs(o["series"]), "pnorm": o["pnorm"], "pulses": _cands(o["pulses"]), "groups": _groups(o["groups"])} for o in outs]


# ---------------------------------------------------------------------------- what a pass cannot do without
def _n_segs(su, dms, t, windows):
    left = [t - int(k) for k in su.shifts(dms).max(1)]
    return [[max(0, (r - int(l)) // max(1, int(l) // 2) + 1) if r >= l else 0 for l in windows] for r in left]


def _fft2(su):
    """Flops of one delay transform by FFTs, and cells of its grid."""
    return 5.0 * su.N * su.Ls * math.log2(su.Ls) + 5.0 * su.Ls * su.Lm * math.log2(su.Lm), float(su.Ls * su.Lm)


def _search_work(su, n_bl, t, dms, windows, sbd_ns):
    """Powers of two: one transform per AP and series, one matrix sum per longer segment; else one transform per
    segment.  Each segment: power and maximum of its cells."""
    fft, cells = _fft2(su)
    if sbd_ns:
        rows = 2 * int(sbd_ns * 1e-3 * 2 * BW) + 1
        fft, cells = fft * min(1.0, rows / su.Ls), cells * min(1.0, rows / su.Ls)
    segs = _n_segs(su, dms, t, windows)
    n = float(sum(map(sum, segs)))
    if all(int(w) & (int(w) - 1) == 0 for w in windows):
        aps = sum(max(0, t - int(k)) for k in su.shifts(dms).max(1))
        longer = sum(s for r in segs for s, w in zip(r, windows) if w > 1)
        flops = aps * fft + longer * 2.0 * cells + n * 3.0 * cells
    else:
        flops = sum(s * (fft + 2.0 * int(w) * su.C) for r in segs for s, w in zip(r, windows)) + n * 3.0 * cells
    slots = sum(max(0, (t - int(w)) // max(1, int(w) // 2) + 1) for w in windows) * len(dms)
    return {"bytes": n_bl * (8.0 * t * su.C + 12.0 * slots), "flops": n_bl * flops}


def work(case):
    do = case["do"]
    if do == "batch":
        dms = np.linspace(0.0, case["dm_hi"], case["n_dm"])
        w = [_search_work(_Setup(s), case["n_bl"], t, dms, (2, 4, 8, 16), 0.0) for s, t in _batch_scans(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    su = _Setup(case["setup"])
    if do == "search":
        return _search_work(su, case["n_bl"], case["t"], np.linspace(0.0, case["dm_hi"], case["n_dm"]), _windows(case), case["sbd_ns"])
    if do == "fit":
        n, fft = case["n_seg"], _fft2(su)
        # mean window 10.5 APs; the points of a segment are read once, no more than the cube holds
        read = min(8.0 * 10.5 * su.C * n, 8.0 * case["n_bl"] * case["t"] * su.C)
        return {"bytes": read + 24.0 * n, "flops": n * (fft[0] + 3.0 * fft[1] + 21.0 * su.C)}
    if do == "refine":
        n = float(case["n_cand"] * case["n_bl"] * int(su.used.sum()))
        # mean width 6.2 APs, three more for the interpolator; about 40 flops a sample forward, 80 backward
        return {"bytes": 8.0 * n * 9.2 + 12.0 * case["n_cand"] * (2 + 3 * case["n_bl"]), "flops": n * 6.2 * 120.0}
    # the calibrator is summed once; per channel a search over 8 J delays
    return {"bytes": 8.0 * case["n_bl"] * case["l"] * su.C + 16.0 * case["n_bl"] * su.N,
            "flops": case["n_bl"] * (2.0 * case["l"] * su.C + su.N * 5.0 * 8 * su.J * math.log2(8 * su.J))}


# ---------------------------------------------------------------------------- 64-bit values
def _dft64(su, dev):
    j, m = torch.arange(su.J, device=dev), torch.arange(su.Ls, device=dev)
    g, q = torch.from_numpy(su.g).to(dev), torch.arange(su.Lm, device=dev)
    es = torch.exp(-2j * math.pi * ((j[:, None] * m[None, :]) % su.Ls).double() / su.Ls)
    em = torch.exp(-2j * math.pi * ((g[:, None] * q[None, :]) % su.Lm).double() / su.Lm)
    return es, em


def _amps64(su, x, rows=None):
    """max |G| over the delay grid of summed spectra x [n][C] (complex128); rows: searched SBD cells."""
    es, em = _dft64(su, x.device)
    if rows is not None:
        es = es[:, rows]
    w = torch.from_numpy(su.used).to(x.device)
    out = torch.empty(x.shape[0], dtype=torch.float64, device=x.device)
    step = max(1, (1 << 24) // (es.shape[1] * su.Lm))
    for i in range(0, x.shape[0], step):
        y = (x[i:i + step] * w).reshape(-1, su.N, su.J) @ es
        gr = y.transpose(1, 2) @ em
        out[i:i + step] = torch.view_as_real(gr).square().sum(-1).flatten(1).amax(1).sqrt()
    return out


def _series64(su, vis, dms, windows, sbd_ns, threads=None):
    """|G| and normalised power of every slot, [n_bl][n_dm][slots]; empty slots -1 and 0."""
    dev = vis.device
    dk = torch.from_numpy(su.shifts(dms)).to(dev)
    rows = None
    if sbd_ns:
        m = np.arange(su.Ls)
        v = np.where(m < su.Ls // 2, m, m - su.Ls) * su.J * 1000.0 / (su.Ls * BW)
        rows = torch.from_numpy(np.flatnonzero(np.abs(v) <= sbd_ns)).to(dev)
    n_bl, t, _ = vis.shape
    off, tot = frbx.frbx_series_layout(t, windows)
    amp = torch.full((n_bl, len(dms), tot), -1.0, dtype=torch.float64, device=dev)
    pn = torch.zeros_like(amp)
    col = torch.arange(su.C, device=dev)
    for b in range(n_bl):
        for d in range(len(dms)):
            kd = t - int(dk[d].max())
            if kd < 1:
                continue
            x = vis[b][torch.arange(kd, device=dev)[:, None] + dk[d][None, :], col[None, :]].to(torch.complex128)
            for l, o in zip(windows, off):
                l, o = int(l), int(o)
                if kd < l:
                    continue
                a = _amps64(su, x.unfold(0, l, max(1, l // 2)).sum(-1), rows)
                amp[b, d, o:o + len(a)] = a
                sd = a.std(correction=0)
                if float(sd) > 0.0:
                    pn[b, d, o:o + len(a)] = (a - a.mean()) / sd
    return amp, pn


def _refine64(su, s):
    p = s["params"].detach().clone().requires_grad_(True)
    vis, t = s["vis"], s["vis"].shape[1]
    n_bl, dev = vis.shape[0], vis.device
    used = torch.from_numpy(np.flatnonzero(su.used)).to(dev)
    f = torch.from_numpy(su.f).to(dev)[used]
    f0 = torch.from_numpy(np.repeat(su.f0, su.J)).to(dev)[used]
    power, width = [], s["width"].tolist()
    grad = torch.zeros_like(p)
    for c in range(p.shape[0]):
        q = p[c].detach().clone().requires_grad_(True)
        u = q[1] + q[0] * (4.15e6 * (1.0 / (f * f) - 1.0 / (su.f.max() * su.f.max())) / su.t_ap)
        x = u[None, :] + torch.arange(width[c], device=dev, dtype=torch.float64)[:, None]
        k = x.detach().floor()
        r = x - k
        w = [0.5 * (-r ** 3 + 2 * r ** 2 - r), 0.5 * (3 * r ** 3 - 5 * r ** 2 + 2), 0.5 * (-3 * r ** 3 + 4 * r ** 2 + r), 0.5 * (r ** 3 - r ** 2)]
        k = k.long()
        ok = ((k >= 1) & (k + 2 <= t - 1)).double()
        tot = 0.0
        for b in range(n_bl):
            smp = sum(w[m] * vis[b][(k - 1 + m).clamp(0, t - 1), used[None, :]].to(torch.complex128) for m in range(4)) * ok
            cyc = ((f - f0) * q[2 + 3 * b] + (f0 - su.f0.min()) * q[3 + 3 * b]) * 1e-3 + f0 * q[4 + 3 * b] * su.t_ap * 1e-6 * x
            gb = (smp * torch.exp(-2j * math.pi * cyc)).sum()
            tot = tot + gb.real ** 2 + gb.imag ** 2
        power.append(tot.detach())
        grad[c], = torch.autograd.grad(tot * s["dpower"][c].double(), q)
    return {"power": torch.stack(power), "grad": grad}


def _calibrate64(su, s):
    vis, dev = s["vis"], s["vis"].device
    used = torch.from_numpy(su.used).to(dev)
    x = torch.stack([v[s["k0"]:s["k0"] + s["l"]].to(torch.complex128).sum(0) for v in vis]) * used
    es, em = _dft64(su, dev)
    g = (x.to(torch.complex64).to(torch.complex128).reshape(-1, su.N, su.J) @ es).transpose(1, 2) @ em
    at = torch.view_as_real(g).square().sum(-1).flatten(1).argmax(1)
    m, q = at // su.Lm, at % su.Lm
    sbd = torch.where(m < su.Ls // 2, m, m - su.Ls).double() * su.J * 1000.0 / (su.Ls * BW)
    mbd = torch.where(q < su.Lm // 2, q, q - su.Lm).double() * 1000.0 / (su.Lm * BW)
    fj = torch.arange(su.J, device=dev, dtype=torch.float64) * BW / su.J
    om = 2 * math.pi * (fj - BW / 2) * 1e-3
    z = x.reshape(-1, su.N, su.J) * torch.exp(-2j * math.pi * fj * 1e-3 * sbd[:, None])[:, None, :]

    def sums(tau):  # D and its first two derivatives at tau [n_bl][N]
        e = z * torch.exp(-1j * om * tau[..., None])
        return e.sum(-1), (-1j * om * e).sum(-1), (-om * om * e).sum(-1)

    n_grid = 8 * su.J
    step = su.J * 1000.0 / (n_grid * BW)
    p = torch.arange(n_grid, device=dev)
    pw = (z @ torch.exp(-1j * om[:, None] * torch.where(p < n_grid // 2, p, p - n_grid).double()[None, :] * step)).abs() ** 2
    kb = pw.argmax(-1, keepdim=True)
    best, lo, hi = (pw.gather(-1, (kb + o) % n_grid).squeeze(-1) for o in (0, -1, 1))
    kb = kb.squeeze(-1)
    tau = (torch.where(kb < n_grid // 2, kb, kb - n_grid).double() + 0.5 * (lo - hi) / (lo - 2 * best + hi)) * step
    for _ in range(8):
        d, d1, d2 = sums(tau)
        f1 = 2 * (d.conj() * d1).real
        f2 = 2 * (d1.abs() ** 2 + (d.conj() * d2).real)
        tau = torch.where(f2 < 0, tau - f1 / f2, tau)
    ph = 2 * math.pi * 1e-3 * (fj * sbd[:, None, None] + torch.from_numpy(su.f0 - su.f0.min()).to(dev)[None, :, None] * mbd[:, None, None]
                               + (fj - BW / 2) * tau[..., None])
    phase = (x.reshape(-1, su.N, su.J) * torch.exp(-1j * ph)).sum(-1).angle()
    return {"sbd": sbd, "mbd": mbd, "delay": tau, "phase": phase}


def exact(case, seed):
    do = case["do"]
    # the direct 64-bit transforms, 8 flops a complex product; about 1e12 of them a second
    def cost(su, segs):
        return segs * 8.0 * (su.C * su.Ls + su.Ls * su.Lm * su.N)
    if do == "batch":
        dms, win = np.linspace(0.0, case["dm_hi"], case["n_dm"]), np.array([2, 4, 8, 16], np.int32)
        if sum(cost(_Setup(n), case["n_bl"] * sum(map(sum, _n_segs(_Setup(n), dms, t, win)))) for n, t in _batch_scans(case)) > 6e12:
            return None
        s = prepare(case, seed)
        out = []
        for (name, _), (_, vis) in zip(_batch_scans(case), s["scans"]):
            amp, pn = _series64(_Setup(name), vis, dms, win, 0.0)
            out.append({"amp": amp, "pnorm": pn})
        return out
    su = _Setup(case["setup"])
    if do == "search":
        dms, win = np.linspace(0.0, case["dm_hi"], case["n_dm"]), _windows(case)
        if cost(su, case["n_bl"] * sum(map(sum, _n_segs(su, dms, case["t"], win)))) > 6e12:
            return None
        s = prepare(case, seed)
        amp, pn = _series64(su, s["vis"].cuda(), dms, win, case["sbd_ns"])
        return {"amp": amp.reshape(-1), "pnorm": pn.reshape(-1)}
    s = prepare(case, seed)
    if do == "fit":
        dk = torch.from_numpy(su.shifts(s["dms"])).cuda()
        col = torch.arange(su.C, device="cuda")
        amp = []
        for i in range(0, len(s["rows"]), 512):
            part = s["rows"][i:i + 512].tolist()
            x = torch.stack([s["vis"][b][k0 + torch.arange(l, device="cuda")[:, None] + dk[d][None, :], col[None, :]].to(torch.complex128).sum(0)
                             for b, d, l, k0 in part])
            amp.append(_amps64(su, x))
        return {"amp": torch.cat(amp)}
    if do == "refine":
        return _refine64(su, s) if case["n_cand"] * case["n_bl"] <= 4000 else None
    return _calibrate64(su, s)
