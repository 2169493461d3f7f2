"""The searches that a user of this library runs, as cases to be measured.

A case is one call, or one short sequence of calls, of the public entry points
(`fstat.Plan(...).search()` / `.set_band()` / `.candidates()` and
`fstat.cell_F_noalloc`) on seeded synthetic data shaped like the narrow-band
segments of the all-sky search.  Plans are made in `prepare`, as a program that
runs many searches makes them; `run` is one search with its read-back.

Thresholds are set as a search sets them, from the false-alarm count that the
grid may return (about 200 noise candidates), and the bands lie at 100 Hz and
above, where an injected signal is found at its own sky position.  The narrow
follow-up ranges keep every F value (threshold below zero).  The FP32 form
computes F in 32 bits and only its record widens it, so those F are returned as
float32; the FP64 form's stay float64.  Candidates are read into an array that the
program keeps (`candidates(cap, out=...)`), which is returned whole.
"""
import math

import numpy as np
import torch

from paper_1410_3677_gb300 import fstat, synth

SPIN_LO = -1e-8          # Hz/s, the spindown range of every grid
DT = 2.0


def _search(name, n, n_sky, n_spin, **more):
    c = {"kind": "search", "n": str(n), "n_fft": 0, "dt": DT, "n_sky": n_sky, "n_spin": n_spin,
         "form": "fp32", "x32": False, "full": False, "interbin": False, "upsample": 2, "frames": 0,
         "bins": 0, "all_bins": False}
    c.update(more)
    if name:
        c["name"] = name
    return c


def _cell(name, n, n_fft):
    c = {"kind": "cell", "n": str(n), "n_fft": n_fft}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # F of one cell into a caller's buffer, from a sky's resampled series: the
        # smallest call there is, all launches and latency
        _cell("cell_2e13", 4096, 8192),
        # the tiny plain grid of the tests and examples: 32 sky x 4 spindowns in FP64
        _search("tiny_fp64", 4096, 32, 4, form="fp64"),
        # short ragged segments in FP32: quick looks at a few hours of data
        _search("short_fp32", 10007, 48, 8, x32=True),
        # the plain FP64 form on the two-sidereal-day segment, one spindown per sky
        # position: reference-precision passes over a sky grid
        _search("sky_fp64", 86164, 192, 1, form="fp64"),
        # a coarse all-sky pass in FP32 with one spindown: the per-sky work counts
        _search("sky_fp32", 86164, 1024, 1),
        # a targeted search: one sky position, many spindowns (the paper's tasks hold 10^4
        # spindowns), three sidereal days
        _search("spins_fp32", 129246, 1, 1024),
        # the main search: consecutive two-sidereal-day frames of one band streamed from
        # pinned host memory through one plan, 64 spindowns per sky position
        _search("frames_fp32", 86164, 256, 64, frames=2),
        # the paper's cheaper transform interpolation on the same grid
        _search("interbin_fp32", 86164, 192, 64, interbin=True),
        # several float32 bands of 1 - 4 sidereal days in one plan
        _search("bands_fp32", "43082,172328,86164,43082,129246", 96, 16, x32=True),
        # the paper's own frame: two sidereal days sampled at 0.5 s (N = 344 656, N_fft = 2^20)
        _search("paper_frame", 344656, 48, 16, dt=0.5),
        # follow-up of one candidate: every F in a narrow frequency range over a fine
        # patch, full JKS statistic, the whole surface read back
        _search("follow_up", 86164, 24, 24, full=True, bins=121),
        # the largest grid listed: one long search of a two-sidereal-day segment
        _search("grid_fp32", 86164, 512, 64),
    ]


# FFT work of the largest listed case, in units of points x log2 points x cells
_MOST = 512 * 64 * 18 * 2.0 ** 18


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One case of the same ranges: segments of 1000 samples to the paper's frame, grids from
    one cell up, both forms, both statistics, both interpolations."""
    what = rng.choice(["cell", "fp64", "fp32", "fp32", "fp32", "fp32", "spins", "interbin", "bands", "follow"])
    if what == "cell":
        n = _log_int(rng, 1500, 131072)
        return _cell(None, n, max(4096, synth.n_fft_auto(n)))
    n = _log_int(rng, 1000, 344656)
    if rng.random() < 0.3:
        n = 43082 * rng.randint(1, 4)           # whole sidereal days
    if what == "follow":
        n = max(n, 22000)
    nf = synth.n_fft_auto(n)
    work = nf * math.log2(nf)
    # the full statistic needs a good part of a sidereal day to tell a(t) from b(t)
    full = n >= 20000 and rng.random() < 0.25
    if what == "fp64":
        cells = max(1.0, min(400.0, 0.004 * _MOST / work))
        n_spin = _log_int(rng, 1, 8)
        return _search(None, n, _log_int(rng, 1, max(1, int(cells / n_spin))), n_spin, form="fp64",
                       full=full)
    more = {"x32": rng.random() < 0.5, "full": full, "upsample": rng.choice([2, 2, 2, 1, 3, 4])}
    if what == "spins":
        return _search(None, n, 1, _log_int(rng, 64, int(min(4096, 0.1 * _MOST / work))), **more)
    if what == "follow":
        n_sky, n_spin = _log_int(rng, 2, 32), _log_int(rng, 2, 32)
        more["full"] = True
        return _search(None, n, n_sky, n_spin, bins=max(17, min(301, int(90000 / (n_sky * n_spin)))), **more)
    if what == "bands":
        more["full"] = False
        ns = [43082 * rng.randint(1, 4) if rng.random() < 0.5 else _log_int(rng, 5000, 172328)
              for _ in range(rng.randint(2, 5))]
        return _search(None, ",".join(str(v) for v in ns), _log_int(rng, 8, 96), _log_int(rng, 4, 24), **more)
    if what == "interbin":
        n = max(n, 2500)
        more["interbin"] = True
    elif rng.random() < 0.2:
        more["all_bins"] = True                 # both halves of the spectrum
    work = 2.0 * synth.n_fft_auto(n) * math.log2(synth.n_fft_auto(n))
    n_spin = _log_int(rng, 1, 128)
    cells = min(8192.0, 0.8 * _MOST / work)
    return _search(None, n, _log_int(rng, 4, max(4, min(2048, int(cells / n_spin)))), n_spin,
                   frames=2 if rng.random() < 0.2 else 0, **more)


# ----------------------------------------------------------------------------- inputs
def _rng(seed, salt):
    return np.random.default_rng([int(seed) & 0x7fffffff, salt])


def _n_fft(case, n):
    return case["n_fft"] or synth.n_fft_auto(n)


def _evals(case):
    tot = 0
    for v in case["n"].split(","):
        nf = _n_fft(case, int(v))
        per = case["bins"] or (nf if case["all_bins"] else nf // 2 - 1)
        tot += case["n_sky"] * case["n_spin"] * per
    return tot


def _threshold(case):
    """2F whose tail (1 + F) e^-F leaves about 200 noise candidates in the grid; the odd bins of
    the interbinned transform carry pi^2/8 of the power.  A follow-up keeps every value."""
    if case["bins"]:
        return -1.0
    t = 8.0
    while _evals(case) * (1.0 + t / 2.0) * math.exp(-t / 2.0) > 200.0:
        t += 0.25
    return t * (1.25 if case["interbin"] else 1.0)


def _grid(case, seed):
    g = _rng(seed, 1)
    n_sky, n_spin = case["n_sky"], case["n_spin"]
    if case["bins"]:                            # a fine patch about one position and spindown
        a0, d0, f0 = g.uniform(0, 2 * math.pi), g.uniform(-1.2, 1.2), g.uniform(-0.9e-8, -0.1e-8)
        alpha = np.mod(a0 + 2e-4 * g.standard_normal(n_sky), 2 * math.pi)
        delta = d0 + 2e-4 * g.standard_normal(n_sky)
        return alpha, delta, f0 + 1e-11 * (np.arange(n_spin) - n_spin // 2)
    if n_sky == 1:                              # a target
        alpha, delta = np.array([g.uniform(0, 2 * math.pi)]), np.array([g.uniform(-1.2, 1.2)])
    else:
        alpha, delta = synth.fibonacci_sky(n_sky)
        alpha = np.mod(alpha + g.uniform(0, 2 * math.pi), 2 * math.pi)
    return alpha, delta, synth.spindown_grid(n_spin, SPIN_LO, 0.0)


def _bands(case, seed):
    """One list of bands per frame (the first for the plan): Gaussian noise and one signal
    on a grid point, a little above the threshold."""
    alpha, delta, fdot = _grid(case, seed)
    frames = []
    for fr in range(max(1, case["frames"])):
        bands = []
        for i, v in enumerate(case["n"].split(",")):
            n, g, edge = int(v), _rng(seed, 100 + 10 * fr + i), _rng(seed, 50 + i)   # frames of a band keep its edge
            nf = _n_fft(case, n)
            sigma = float(g.uniform(0.5, 2.0))
            t = max(_threshold(case), 40.0)
            inj = synth.draw_injections(g, 1, alpha.size, fdot.size, nf, case["dt"], math.sqrt(t + 15.0),
                                        math.sqrt(t + 45.0), 0.05 / case["dt"], 0.45 / case["dt"])
            bands.append(synth.make_band(n, case["dt"], int(g.integers(1 << 30)), sigma, alpha, delta, fdot, inj,
                                         f_off=100.0 + (1.0 - 2.0 ** -5) * (i + int(edge.integers(32))), n_fft=nf,
                                         dtype=np.float32 if case["x32"] else np.float64))
        frames.append(bands)
    return alpha, delta, fdot, frames


def _bin_range(case, seed):
    if case["bins"]:
        nf = _n_fft(case, int(case["n"]))
        lo = int(_rng(seed, 2).integers(nf // 16, nf // 2 - 512 - case["bins"]) if nf >= 4096 else nf // 8)
        return lo, lo + case["bins"] - 1
    if case["all_bins"]:
        return 0, min(_n_fft(case, int(v)) for v in case["n"].split(",")) - 1
    return 0, 0                                 # the default: 1 .. n_fft / 2 - 1


def _pinned(a):
    return torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()


def _cell_inputs(case, seed):
    """A sky's demodulated series (y a, y b), the tail outside the resampling window zero, and a
    spindown rate and normalisers as a search of two days' data has them."""
    n, g = int(case["n"]), _rng(seed, 3)
    t = np.arange(n) * DT
    y = g.standard_normal(n) * np.exp(-2j * np.pi * np.mod(g.uniform(100, 130) * 300 * np.sin(2e-7 * t + 1), 1.0))
    y[n - n // 40:] = 0.0
    a = 0.4 + 0.5 * np.cos(1.4584e-4 * t + g.uniform(0, 6)) + 0.2 * np.sin(7.292e-5 * t)
    b = 0.6 * np.sin(1.4584e-4 * t + g.uniform(0, 6)) - 0.2 * np.cos(7.292e-5 * t)
    w = np.stack([(y * a).real, (y * a).imag, (y * b).real, (y * b).imag], axis=1).astype(np.float32)
    return w, float(0.5 * g.uniform(SPIN_LO, 0.0) * DT * DT), float(1.0 / np.sum(a * a)), float(1.0 / np.sum(b * b))


# ----------------------------------------------------------------------------- the path
def prepare(case, seed):
    if case["kind"] == "cell":
        w, rate, na, nb = _cell_inputs(case, seed)
        nf = case["n_fft"]
        return {"kind": "cell", "w": torch.from_numpy(w).cuda(), "n": int(case["n"]), "n_fft": nf, "rate": rate,
                "na": na, "nb": nb, "F": torch.zeros(nf // 2 - 1, dtype=torch.float32, device="cuda")}
    alpha, delta, fdot, frames = _bands(case, seed)
    lo, hi = _bin_range(case, seed)
    fp64 = case["form"] == "fp64"
    plan = fstat.Plan(frames[0], alpha, delta, fdot, _threshold(case), lat=synth.LAT_DEFAULT,
                      gamma=synth.GAMMA_DEFAULT, upsample=case["upsample"],
                      form=fstat.FP64_PLAIN if fp64 else fstat.FP32_BATCHED, bin_lo=lo, bin_hi=hi,
                      cand_capacity=1 << 20, full=case["full"], interbin=case["interbin"])
    segments = []
    for bands in frames if case["frames"] else []:
        for b in bands:
            b.x, b.r = _pinned(b.x), _pinned(b.r)
        segments.append(bands[0])
    return {"kind": "search", "plan": plan, "segments": segments, "fp64": fp64,
            "found": [np.zeros(_room(case), fstat.CAND_DTYPE) for _ in frames]}


def _room(case):
    """Records a program makes room for: every value of a follow-up, else a few times the
    expected candidates."""
    return case["n_sky"] * case["n_spin"] * case["bins"] if case["bins"] else 4096


def _records(c, total, fp64):
    out = {k: c[k] for k in ("band", "sky", "spin", "bin", "alpha", "delta", "freq", "fdot")}
    out["F"] = c["F"] if fp64 else c["F"].astype(np.float32)
    out["total"] = total
    return out


def run(state):
    if state["kind"] == "cell":
        F = state["F"]
        rc = fstat.cell_F_noalloc(state["w"].data_ptr(), state["n"], state["n_fft"], state["rate"], state["na"],
                                  state["nb"], 1, state["n_fft"] // 2 - 1, F.data_ptr())
        if rc != fstat.FSTAT_OK:
            raise RuntimeError(fstat.status_string(rc))
        return F
    plan, out = state["plan"], []
    for i, buf in enumerate(state["found"]):
        if state["segments"]:
            plan.set_band(0, state["segments"][i])   # the next frame of the band
        plan.search()
        _, total = plan.candidates(buf.size, out=buf)
        out.append(_records(buf, total, state["fp64"]))
    return out


# ----------------------------------------------------------------------------- its work
def work(case):
    """Bytes: each series and ephemeris once, each returned value once.  FLOPs: two transforms
    per cell, 5 N log2 N each (half the length when interbinning)."""
    if case["kind"] == "cell":
        n, nf = int(case["n"]), case["n_fft"]
        return {"bytes": 16.0 * n + 4.0 * (nf // 2 - 1), "flops": 10.0 * nf * math.log2(nf)}
    cells, b, f = case["n_sky"] * case["n_spin"], 0.0, 0.0
    for v in case["n"].split(","):
        n, nf = int(v), _n_fft(case, int(v))
        t = nf // 2 if case["interbin"] else nf
        b += n * ((4.0 if case["x32"] else 8.0) + 24.0)
        f += cells * 10.0 * t * math.log2(t)
    b += 72.0 * _room(case)
    k = max(1, case["frames"])
    return {"bytes": k * b, "flops": k * f}


# ----------------------------------------------------------------------------- 64-bit values
def _delay_at(d, u):
    n = d.numel()
    j = torch.floor(u).clamp(0, n - 2).long()
    return d[j] + (u - j) * (d[j + 1] - d[j])


def _upsampled(x, U):
    n = x.numel()
    X = torch.fft.fft(x.to(torch.complex128))
    m = torch.arange(n, device=x.device, dtype=torch.int64)
    m = torch.where(2 * m < n, m, m - n)
    out = torch.empty(n, U, dtype=torch.float64, device=x.device)
    out[:, 0] = x
    for s in range(1, U):
        ph = 2 * math.pi * torch.remainder(m * s, U * n).double() / (U * n)
        Y = X * torch.polar(torch.ones_like(ph), ph)
        if n % 2 == 0:
            Y[n // 2] = X[n // 2] * math.cos(math.pi * s / U)
        out[:, s] = torch.fft.ifft(Y).real
    return out.reshape(-1)


def _sky_series(x, xu, U, r, band, al, de):
    """(y a, y b) of one sky position and the sums of a^2, b^2, a b over the resampling window."""
    n, dt = x.numel(), band.dt
    k = torch.arange(n, device=x.device, dtype=torch.float64)
    nh = torch.tensor([math.cos(de) * math.cos(al), math.cos(de) * math.sin(al), math.sin(de)],
                      dtype=torch.float64, device=x.device)
    d = r @ nh
    u = k - _delay_at(d, k - d / dt) / dt
    ok = (u >= 0) & (u <= n - 1)
    p = U * u
    pf = torch.floor(p)
    mu, i0 = p - pf, pf.long() - 1
    tap = [xu[torch.remainder(i0 + q, U * n)] for q in range(4)]
    v = (((-0.5 * mu + 1.0) * mu - 0.5) * mu * tap[0] + ((1.5 * mu - 2.5) * mu * mu + 1.0) * tap[1]
         + ((-1.5 * mu + 2.0) * mu + 0.5) * mu * tap[2] + (0.5 * mu - 0.5) * mu * mu * tap[3])
    cyc = band.f_off * _delay_at(d, u)
    y = torch.where(ok, v, torch.zeros_like(v)) * torch.polar(torch.ones_like(v), -2 * math.pi * (cyc - torch.floor(cyc)))
    h = al - (band.phi0 + synth.OMEGA_R * u * dt)
    lat, gam = synth.LAT_DEFAULT, synth.GAMMA_DEFAULT
    s2g, c2g = math.sin(2 * gam), math.cos(2 * gam)
    c1, s1, c2, s2 = torch.cos(h), torch.sin(h), torch.cos(2 * h), torch.sin(2 * h)
    a = (s2g * (3 - math.cos(2 * lat)) * (3 - math.cos(2 * de)) / 16 * c2 - c2g * math.sin(lat) * (3 - math.cos(2 * de)) / 4 * s2
         + s2g * math.sin(2 * lat) * math.sin(2 * de) / 4 * c1 - c2g * math.cos(lat) * math.sin(2 * de) / 2 * s1
         + 0.75 * s2g * math.cos(lat) ** 2 * math.cos(de) ** 2)
    b = (c2g * math.sin(lat) * math.sin(de) * c2 + s2g * (3 - math.cos(2 * lat)) * math.sin(de) / 4 * s2
         + c2g * math.cos(lat) * math.cos(de) * c1 + s2g * math.sin(2 * lat) * math.cos(de) / 2 * s1)
    a, b = torch.where(ok, a, 0 * a), torch.where(ok, b, 0 * b)
    return torch.stack([y * a, y * b]), float((a * a).sum()), float((b * b).sum()), float((a * b).sum())


def _exact_search(case, seed):
    alpha, delta, fdot, frames = _bands(case, seed)
    lo0, hi0 = _bin_range(case, seed)
    thr, U = _threshold(case), case["upsample"]
    found = []
    for bands in frames:
        rows = {q: [] for q in ("band", "sky", "spin", "bin", "F")}
        for bi, band in enumerate(bands):
            x = torch.from_numpy(band.x.astype(np.float64)).cuda()
            r = torch.from_numpy(band.r).cuda()
            n, nf = band.n, band.n_fft
            lo, hi = (lo0, hi0) if (lo0 or hi0) else (1, nf // 2 - 1)
            xu = _upsampled(x, U)
            s2 = float((x * x).mean())
            k2 = torch.arange(n, device="cuda", dtype=torch.float64) ** 2
            rate = torch.from_numpy(0.5 * fdot * band.dt * band.dt).cuda()
            step = max(1, int(2 ** 27 // (2 * nf)))
            for si in range(alpha.size):
                w, Saa, Sbb, Sab = _sky_series(x, xu, U, r, band, float(alpha[si]), float(delta[si]))
                if case["full"]:
                    D = Saa * Sbb - Sab * Sab
                    na, nb, nab = Sbb / (s2 * D), Saa / (s2 * D), -2.0 * Sab / (s2 * D)
                else:
                    na, nb, nab = 1.0 / (s2 * Saa), 1.0 / (s2 * Sbb), 0.0
                for j0 in range(0, fdot.size, step):
                    cyc = rate[j0:j0 + step, None] * k2[None, :]
                    ph = -2 * math.pi * (cyc - torch.floor(cyc))
                    z = w[None] * torch.polar(torch.ones_like(ph), ph)[:, None, :]
                    if case["interbin"]:
                        X = torch.fft.fft(z, n=nf // 2)
                        odd = (math.pi / 4) * (X - torch.roll(X, -1, dims=-1))
                        X = torch.stack([X, odd], dim=-1).reshape(z.shape[0], 2, nf)
                    else:
                        X = torch.fft.fft(z, n=nf)
                    A, B = X[:, 0, lo:hi + 1], X[:, 1, lo:hi + 1]
                    F = (A.real ** 2 + A.imag ** 2) * na + (B.real ** 2 + B.imag ** 2) * nb
                    if nab:
                        F = F + (A.real * B.real + A.imag * B.imag) * nab
                    hit = torch.nonzero(2 * F > thr)
                    rows["F"].append(F[hit[:, 0], hit[:, 1]].cpu().numpy())
                    hit = hit.cpu().numpy()
                    rows["spin"].append(hit[:, 0] + j0)
                    rows["bin"].append(hit[:, 1] + lo)
                    rows["sky"].append(np.full(len(hit), si))
                    rows["band"].append(np.full(len(hit), bi))
        o = {q: np.concatenate(v) for q, v in rows.items()}
        o["alpha"], o["delta"], o["fdot"] = alpha[o["sky"]], delta[o["sky"]], fdot[o["spin"]]
        f_off, df = (np.array([v(b) for b in bands]) for v in (lambda b: b.f_off, lambda b: b.n_fft * b.dt))
        o["freq"] = f_off[o["band"]] + o["bin"] / df[o["band"]]
        room = _room(case)                      # in the order of the read-back, the rest of the array zero
        o = {q: np.concatenate([v[:room], np.zeros(max(0, room - len(v)), v.dtype)]) for q, v in o.items()}
        found.append(dict(o, total=sum(len(v) for v in rows["F"])))
    return found


def exact(case, seed):
    if case["kind"] == "search":
        return _exact_search(case, seed)
    w, rate, na, nb = _cell_inputs(case, seed)
    w = torch.view_as_complex(torch.from_numpy(w.astype(np.float64)).cuda().reshape(-1, 2, 2))
    cyc = rate * torch.arange(int(case["n"]), device="cuda", dtype=torch.float64) ** 2
    ph = -2 * math.pi * (cyc - torch.floor(cyc))
    X = torch.fft.fft(w * torch.polar(torch.ones_like(ph), ph)[:, None], n=case["n_fft"], dim=0)[1:case["n_fft"] // 2]
    return (X[:, 0].real ** 2 + X[:, 0].imag ** 2) * na + (X[:, 1].real ** 2 + X[:, 1].imag ** 2) * nb
