"""What this library is timed on: the calls an imaging or search program makes,
over the sizes it makes them at.

Every case goes through the Python binding of the C ABI
(`paper_2301_09662_gb300.epic`): `Plan.image`, `Plan.image_series`,
`Plan.image_efield`, `Plan.solve_gains`, and `Search.dedisperse` with
`Search.single_pulse`.  The shapes are those of `synth` and `bench.py`: the
16-antenna tiny array, the 256-antenna LWA-like station (64 channels, 128 x 128
grids, 1000 spectra of 40 us), its 30-80 MHz band with three grid sides, and
the 2048-antenna dense array (512 x 512 grids).

Voltages are complex Gaussian noise (sigma 2 per component) plus three point
sources seen through the array's geometry, rounded to 4+4 bits, as from an
F-engine; layouts, gains and delays come from the same seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2301_09662_gb300 import epic, synth

C0 = 299_792_458.0
K_DM = 4.148808e3                       # s MHz^2 pc^-1 cm^3
WIDTHS = (1, 2, 4, 8, 16, 32)
PRECISION = {"fp32": epic.EPIC_FP32, "split_fp16": epic.EPIC_TC_SPLIT_FP16, "fp16": epic.EPIC_TC_FP16}


def _imaging(name, what, precision, A, P, C, T, sides, K, f0, f1, diam_x, diam_y, spacing=0.0, gains=True,
             taper=False, stokes=False, delays=False, antenna_kernels=False, spi=0):
    """sides: grid sides, e.g. "128", or "64/96/128" for that many equal blocks of channels."""
    return {"name": name, "what": what, "precision": precision, "A": A, "P": P, "C": C, "T": T, "sides": sides,
            "K": K, "f0": float(f0), "f1": float(f1), "diam_x": float(diam_x), "diam_y": float(diam_y),
            "spacing": float(spacing), "gains": gains, "taper": taper, "stokes": stokes, "delays": delays,
            "antenna_kernels": antenna_kernels, "spi": spi}


def listed():
    station = dict(A=256, P=2, C=64, K=5, f0=60e6, f1=61.575e6, diam_x=110, diam_y=100, spacing=4.0)
    return [
        # the smallest call: a handful of single-polarisation antennas, one short integration; the
        # time is launches and latency
        _imaging("tiny_fp32", "image", "fp32", A=16, P=1, C=4, T=64, sides="32", K=3, f0=40e6, f1=40.75e6,
                 diam_x=40, diam_y=40, gains=False),
        # a narrow slice of the station imaged every 64 spectra, kernel applied as an image taper:
        # short calls of a transient monitor
        _imaging("short_taper_fp32", "image", "fp32", T=64, sides="128", taper=True, **{**station, "C": 16}),
        # the station's normal product: one 40 ms integration of 64 channels, calibrated, four
        # polarisation products, in the FP32 form and in the tensor-core form
        _imaging("station_fp32", "image", "fp32", T=1000, sides="128", **station),
        _imaging("station_split_fp16", "image", "split_fp16", T=1000, sides="128", **station),
        # the whole 30-80 MHz band, grid side following frequency, tensor-core form
        _imaging("band_split_fp16", "image", "split_fp16", A=256, P=2, C=192, T=1000, sides="64/96/128", K=5,
                 f0=30e6, f1=80e6, diam_x=110, diam_y=100, spacing=4.0),
        # odd sizes: a partly populated station, 37 channels over the same band, a ragged integration
        _imaging("ragged_band_fp32", "image", "fp32", A=202, P=2, C=37, T=333, sides="64/96/128", K=3,
                 f0=30e6, f1=80e6, diam_x=110, diam_y=100, spacing=4.0),
        # the dense array: many antennas, wide kernel, large grids
        _imaging("dense_fp32", "image", "fp32", A=2048, P=2, C=64, T=100, sides="512", K=7, f0=49e6, f1=50.575e6,
                 diam_x=350, diam_y=350, spacing=3.0),
        # millisecond imaging: Stokes images of 40 spectra each from one integration, with the
        # geometric delays of a drifting phase centre
        _imaging("series_stokes_fp32", "series", "fp32", T=1000, sides="128", stokes=True, delays=True, spi=40,
                 **station),
        # electric-field images of every sample (what a beamformer or a polarimeter taps)
        _imaging("efield_fp32", "efield", "fp32", T=50, sides="128", **station),
        # A-projection: every antenna with its own illumination kernel
        _imaging("antenna_kernels_fp32", "image", "fp32", T=250, sides="128", antenna_kernels=True, **station),
        # transient search of an image cube: 128 trial DMs and the single-pulse search of every
        # de-dispersed light curve
        {"name": "search_cube", "what": "search", "C": 72, "n_pix": 4096, "n_time": 512, "n_dm": 128,
         "dm_max": 25.4, "f0": 42.1e6, "df": 25e3, "dt": 0.04},
        # gain solution from one calibrator over a whole integration
        _imaging("solve_gains", "gains", "fp32", T=1000, sides="128", **station),
    ]


def draw(rng):
    """One more case of the listed ranges."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["image"] * 6 + ["series", "efield", "gains", "search", "dense"])
    if what == "search":
        C, npix, nt, ndm = logint(8, 96), logint(64, 4096), logint(96, 512), logint(4, 128)
        # the largest sweep stays below half of the series
        f0, df, dt = rng.choice([42.1e6, 60e6, 72.3e6]), 25e3, rng.choice([0.005, 0.04])
        top = (f0 + (C - 1) * df) / 1e6
        per_dm = K_DM * ((f0 / 1e6) ** -2 - top ** -2) / dt
        dm_max = rng.uniform(0.2, 1.0) * min(30.0, 0.45 * nt / per_dm)
        return {"what": "search", "C": C, "n_pix": npix, "n_time": nt, "n_dm": ndm, "dm_max": dm_max, "f0": f0,
                "df": df, "dt": dt}
    if what == "dense":
        A, K = logint(300, 2048), rng.choice([5, 7])
        side = rng.choice(["256", "512"])
        C, T = logint(2, 32), logint(16, 100)
        diam = rng.uniform(0.5, 1.0) * (int(side) / 2 - K - 2) * 0.5 * C0 / 51e6
        return _imaging("", "image", "fp32", A=A & ~1, P=2, C=C, T=T, sides=side, K=K, f0=49e6, f1=50.5e6,
                        diam_x=diam, diam_y=diam, gains=rng.random() < 0.8)
    precision = rng.choice(["fp32", "fp32", "split_fp16", "fp16"]) if what in ("image", "series") else "fp32"
    P = 2 if precision != "fp32" else rng.choice([1, 2, 2, 2])
    A = logint(16, 512) if what != "series" and precision == "fp32" else logint(16, 256)
    if precision != "fp32" or what == "efield":
        A = max(16, A & ~3)
    K = rng.choice([1, 3, 5, 7])
    if precision != "fp32" and K == 7:
        A = min(A, 128)
    sides = rng.choice(["64", "96", "128", "128", "64/96/128"])
    if precision == "fp32" and what in ("image", "gains") and rng.random() < 0.2:
        sides = "32"
    C = logint(3, 64)
    T = logint(8, 1000) if what != "efield" else logint(4, 50)
    f0 = rng.uniform(30e6, 70e6)
    f1 = f0 + 25e3 * (C - 1) if "/" not in sides else f0 + rng.uniform(2e6, 10e6)
    smallest = min(int(s) for s in sides.split("/"))
    diam = rng.uniform(0.4, 1.0) * max(4.0, smallest / 2 - K - 2) * 0.5 * C0 / f1
    spi = 0
    if what == "series":
        spi = logint(8, 100)
        T = spi * logint(1, max(1, min(25, 1000 // spi)))
    plain = what == "image" and precision == "fp32"
    kernels = plain and K > 1 and A <= 256 and rng.random() < 0.15
    return _imaging("", what, precision, A=A, P=P, C=C, T=T, sides=sides, K=K, f0=f0, f1=f1, diam_x=diam,
                    diam_y=diam * rng.uniform(0.8, 1.0), gains=rng.random() < 0.8,
                    taper=what == "image" and not kernels and rng.random() < 0.2,
                    stokes=P == 2 and what in ("image", "series") and rng.random() < 0.3,
                    delays=what in ("image", "series") and not kernels and rng.random() < 0.25,
                    antenna_kernels=kernels, spi=spi)


# ---------------------------------------------------------------- inputs

def _grid_sides(case):
    s = [int(x) for x in case["sides"].split("/")]
    C = case["C"]
    return np.array([s[min(len(s) - 1, c * len(s) // C)] for c in range(C)], np.int32)


def _inputs(case, seed):
    """Geometry (numpy) and device tensors of an imaging case."""
    rng = np.random.default_rng([seed, 20230120])
    A, P, C, T, K = case["A"], case["P"], case["C"], case["T"], case["K"]
    ant = synth.layout_ellipse(A, case["diam_x"] / 2, case["diam_y"] / 2, rng, case["spacing"])
    freq = np.linspace(case["f0"], case["f1"], C)
    kern = synth.antenna_kernels(A, K, rng) if case["antenna_kernels"] else synth.gaussian_kernel(K)
    gains = torch.from_numpy(synth.random_gains(C, A, P, rng)).cuda() if case["gains"] else None
    delays = torch.from_numpy(synth.geometric_delays(ant, T, l0=rng.uniform(-0.4, 0.4))).cuda() \
        if case["delays"] else None
    calibrator = rng.uniform(-0.4, 0.4, 2)
    lm = rng.uniform(-0.5, 0.5, (3, 2))
    flux = [1.0, 0.3, 0.1]
    if case["what"] == "gains":            # the calibrator dominates its field
        lm[0] = calibrator
        flux = [9.0, 0.3, 0.1]
    gen = torch.Generator("cuda").manual_seed(seed)
    v = torch.empty((T, C, A, P), dtype=torch.uint8, device="cuda")
    uv = (ant - ant.mean(axis=0))[None] * (freq[:, None, None] / C0)              # [C][A][2] wavelengths
    for t0 in range(0, T, 100):
        n = min(100, T - t0)
        re = torch.randn((n, C, A, P), generator=gen, device="cuda") * 2.0
        im = torch.randn((n, C, A, P), generator=gen, device="cuda") * 2.0
        for s in range(3):
            ph = -2.0 * np.pi * (uv @ lm[s])
            pr = torch.from_numpy(np.cos(ph).astype(np.float32)).cuda()[None, :, :, None]
            pi = torch.from_numpy(np.sin(ph).astype(np.float32)).cuda()[None, :, :, None]
            z = torch.randn((2, n, C, 1, P), generator=gen, device="cuda") * math.sqrt(flux[s] / 2.0)
            re += z[0] * pr - z[1] * pi
            im += z[0] * pi + z[1] * pr
        re = torch.round(re).clamp_(-7, 7).to(torch.int32)
        im = torch.round(im).clamp_(-7, 7).to(torch.int32)
        v[t0:t0 + n] = (((re & 15) << 4) | (im & 15)).to(torch.uint8)
    return {"ant": ant, "freq": freq, "kern": kern, "grid": _grid_sides(case), "v": v, "gains": gains,
            "delays": delays, "calibrator": calibrator}


def _search_inputs(case, seed):
    """Intensity cube [T][C][pixels]: Gaussian noise and a few dispersed pulses."""
    rng = np.random.default_rng([seed, 20230121])
    C, npix, T = case["C"], case["n_pix"], case["n_time"]
    freq = case["f0"] + case["df"] * np.arange(C)
    dms = np.linspace(0.0, case["dm_max"], case["n_dm"])
    gen = torch.Generator("cuda").manual_seed(seed)
    cube = torch.randn((T, C, npix), generator=gen, device="cuda") + 10.0
    shifts = _dm_shifts(freq, case["dt"], dms)
    for _ in range(12):
        d, p, t = int(rng.integers(len(dms))), int(rng.integers(npix)), int(rng.integers(T - shifts.max()))
        amp = float(rng.uniform(0.5, 3.0))
        idx = torch.from_numpy(np.minimum(t + shifts[d], T - 1)).cuda()
        cube[idx, torch.arange(C, device="cuda"), p] += amp
    return freq, dms, cube


def _dm_shifts(freq, dt, dms):
    f = np.asarray(freq) / 1e6
    return np.floor(K_DM * dms[:, None] * (f[None] ** -2 - f.max() ** -2) / dt + 0.5).astype(np.int64)


def prepare(case, seed):
    """The plan, the device-resident inputs and the output buffers a program keeps."""
    if case["what"] == "search":
        freq, dms, cube = _search_inputs(case, seed)
        s = epic.Search(freq, case["dt"], dms, case["n_pix"], case["n_time"], widths=_widths(case, freq, dms))
        dd = torch.empty((s.n_dm, s.t_out, s.n_pix), dtype=torch.float32, device="cuda")
        return {"what": "search", "search": s, "cube": cube, "dd": dd}
    x = _inputs(case, seed)
    flags = (epic.EPIC_KERNEL_TAPER if case["taper"] else 0) | (epic.EPIC_STOKES if case["stokes"] else 0) | \
        (epic.EPIC_ANTENNA_KERNELS if case["antenna_kernels"] else 0)
    plan = epic.Plan(x["ant"], case["P"], x["kern"], x["grid"], x["freq"], 0.5, case["T"],
                     PRECISION[case["precision"]], flags)
    n = plan.out_floats // 2
    T = case["T"]
    shape = {"image": (n,), "series": (T // case["spi"] if case["spi"] else 0, n), "gains": (plan.C, plan.A, plan.P),
             "efield": (T, int(case["P"] * np.sum(x["grid"].astype(np.int64) ** 2)))}[case["what"]]
    out = torch.empty(shape, dtype=torch.complex64, device="cuda")
    return {"what": case["what"], "plan": plan, "v": x["v"], "gains": x["gains"], "delays": x["delays"], "out": out,
            "spi": case["spi"], "calibrator": x["calibrator"]}


def _widths(case, freq, dms):
    t_out = case["n_time"] - int(_dm_shifts(freq, case["dt"], dms).max())
    return tuple(w for w in WIDTHS if w <= t_out)


def run(state):
    what = state["what"]
    if what == "search":
        s = state["search"]
        dd = s.dedisperse(state["cube"], out=state["dd"])
        # the candidate list is undefined past its count, so the count stands for it here
        snr, t, w, _, n = s.single_pulse(dd, 6.0)
        return {"dd": dd, "snr": snr, "t": t, "w": w, "n": n}
    plan = state["plan"]
    if what == "image":
        return plan.image(state["v"], state["gains"], out=state["out"], delays=state["delays"])
    if what == "series":
        return plan.image_series(state["v"], state["spi"], state["gains"], out=state["out"], delays=state["delays"])
    if what == "efield":
        return plan.image_efield(state["v"], state["gains"], out=state["out"])
    l, m = state["calibrator"]
    return plan.solve_gains(state["v"], l, m, 2, out=state["out"])


# ---------------------------------------------------------------- floors and tolerances

def work(case):
    """Inputs read once, results written once; the arithmetic of the plain method: gridding
    8 A K^2, a radix-2 transform of the occupied half of the rows and of every column, 8 N^2 for
    the products of each spectrum."""
    if case["what"] == "search":
        freq = case["f0"] + case["df"] * np.arange(case["C"])
        dms = np.linspace(0.0, case["dm_max"], case["n_dm"])
        t_out = case["n_time"] - int(_dm_shifts(freq, case["dt"], dms).max())
        nd = case["n_dm"] * t_out * case["n_pix"]
        pairs = case["n_dm"] * case["n_pix"]
        return {"bytes": 4 * (case["n_time"] * case["C"] * case["n_pix"] + nd + 3 * pairs),
                "flops": nd * (case["C"] + 5 + 3)}
    A, P, C, T = case["A"], case["P"], case["C"], case["T"]
    n2 = int(np.sum(_grid_sides(case).astype(np.int64) ** 2))
    b = T * C * A * P + (8 * C * A * P if case["gains"] else 0) + (8 * T * A if case["delays"] else 0)
    if case["what"] == "gains":
        return {"bytes": b + 8 * C * A * P, "flops": 2 * 2 * 8 * T * C * A * P}
    K2 = 1 if case["taper"] else case["K"] ** 2
    flops = 0
    for N in _grid_sides(case):
        N = int(N)
        flops += T * P * (8 * A * K2 + 5 * N * math.log2(N) * (N / 2 + N) + (8 * N * N if case["what"] != "efield" else 0))
    images = {"image": 1, "series": T // case["spi"] if case["spi"] else 1, "efield": T}[case["what"]]
    planes = P if case["what"] == "efield" else (4 if P == 2 else 1)
    return {"bytes": b + 8 * planes * n2 * images, "flops": int(flops)}


def tolerance(case):
    """About four times the error measured against the 64-bit results (2-norm: FP32 images 1.9e-6,
    E-field images 1.3e-7, split FP16 1.5e-5, FP16 1.2e-3, gains 7e-7, S/N 3.4e-6; largest
    difference over the root mean square: FP32 8e-5, split FP16 1e-4, FP16 2.2e-2)."""
    if case["what"] == "search":
        return {"rel": 1e-5, "max": 1e-4, "differ": 1e-4}   # best windows tie within a rounding of S/N
    if case["what"] == "gains":
        return {"rel": 3e-6, "max": 3e-5}
    if case["what"] == "efield":
        return {"rel": 1e-6, "max": 1e-5}
    if case["precision"] == "fp16":
        return {"rel": 5e-3, "max": 1e-1}     # 11-bit operands
    if case["precision"] == "split_fp16":
        return {"rel": 6e-5, "max": 6e-4}
    return {"rel": 8e-6, "max": 3e-4}


# ---------------------------------------------------------------- the same results in 64 bits

def _decode(v):
    re = (v >> 4).to(torch.float64)
    im = (v & 15).to(torch.float64)
    re = torch.where(re > 7, re - 16, re)
    im = torch.where(im > 7, im - 16, im)
    return torch.complex(re, im)


def _cells(ant, freq, N):
    d = ant - ant.mean(axis=0)
    x = d * freq / (C0 * 0.5)
    return (np.sign(x) * np.floor(np.abs(x) + 0.5)).astype(np.int64) + N // 2     # [A][2]


def _fields(x, case, c, t0, t1):
    """Electric fields [t][P][N][N] of one channel, shifted, and the calibrated voltages [t][P][A]."""
    N, K = int(x["grid"][c]), case["K"]
    h = (K - 1) // 2
    e = _decode(x["v"][t0:t1, c]).permute(0, 2, 1)                              # [t][P][A]
    if x["gains"] is not None:
        e = e * x["gains"][c].to(torch.complex128).T[None]
    if x["delays"] is not None:
        ph = 2.0 * math.pi * torch.remainder(x["delays"][t0:t1] * x["freq"][c], 1.0)
        e = e * torch.polar(torch.ones_like(ph), ph)[:, None, :]
    k = _cells(x["ant"], x["freq"][c], N)
    n, P = t1 - t0, case["P"]
    grid = torch.zeros((n * P, N * N), dtype=torch.complex128, device="cuda")
    flat = e.reshape(n * P, -1)
    w = torch.from_numpy(x["kern"].astype(np.complex128)).cuda()
    for dy in range(-h, h + 1):
        for dx in range(-h, h + 1):
            at = torch.from_numpy((k[:, 1] + dy) * N + k[:, 0] + dx).cuda()
            grid.index_add_(1, at, flat * w[..., dy + h, dx + h])
    F = torch.fft.ifft2(grid.view(n, P, N, N), norm="forward")
    return torch.fft.fftshift(F, dim=(2, 3)), e


def _kernel_power(w, N):
    K = w.shape[-1]
    g = torch.zeros(w.shape[:-2] + (N, N), dtype=torch.complex128, device="cuda")
    g[..., :K, :K] = w
    return torch.fft.fftshift(torch.fft.ifft2(g, norm="forward").abs() ** 2, dim=(-2, -1))


def _image(x, case, c, t0, t1):
    """[NP][N][N] image of channel c over spectra t0 .. t1, autocorrelations subtracted."""
    N, P = int(x["grid"][c]), case["P"]
    step = max(1, (1 << 25) // (P * N * N))
    S = torch.zeros((3, N, N), dtype=torch.complex128, device="cuda")
    auto = torch.zeros((3, case["A"]), dtype=torch.complex128, device="cuda")
    for a in range(t0, t1, step):
        F, e = _fields(x, case, c, a, min(t1, a + step))
        S[0] += (F[:, 0].abs() ** 2).sum(0)
        auto[0] += (e[:, 0].abs() ** 2).sum(0)
        if P == 2:
            S[1] += (F[:, 1].abs() ** 2).sum(0)
            S[2] += (F[:, 0] * F[:, 1].conj()).sum(0)
            auto[1] += (e[:, 1].abs() ** 2).sum(0)
            auto[2] += (e[:, 0] * e[:, 1].conj()).sum(0)
    w = torch.from_numpy(x["kern"].astype(np.complex128)).cuda()
    power = _kernel_power(w, N).to(torch.complex128)
    if case["antenna_kernels"]:
        S -= (auto @ power.view(case["A"], N * N)).view(3, N, N)
    else:
        S -= auto.sum(1)[:, None, None] * power[None]
    if P == 1:
        return S[:1]
    if case["stokes"]:
        zero = torch.zeros_like(S[0].real)
        return torch.stack([torch.complex(s, zero) for s in
                            (S[0].real + S[1].real, S[0].real - S[1].real, 2 * S[2].real, 2 * S[2].imag)])
    return torch.stack([S[0], S[1], S[2], S[2].conj()])


def _exact_search(case, seed):
    freq, dms, cube = _search_inputs(case, seed)
    shifts = _dm_shifts(freq, case["dt"], dms)
    widths = _widths(case, freq, dms)
    T_out = case["n_time"] - int(shifts.max())
    npix = case["n_pix"]
    dd = torch.empty((len(dms), T_out, npix), dtype=torch.float64, device="cuda")
    snr = torch.empty((len(dms), npix), dtype=torch.float64, device="cuda")
    bt = torch.empty((len(dms), npix), dtype=torch.int32, device="cuda")
    bw = torch.empty_like(bt)
    for d in range(len(dms)):
        acc = torch.zeros((T_out, npix), dtype=torch.float64, device="cuda")
        for c in range(case["C"]):
            s = int(shifts[d, c])
            acc += cube[s:s + T_out, c].double()
        dd[d] = acc
        mu, sigma = acc.mean(0), acc.std(0, unbiased=False)
        cum = torch.cat([torch.zeros((1, npix), dtype=torch.float64, device="cuda"), (acc - mu).cumsum(0)])
        best = torch.full((npix,), -math.inf, dtype=torch.float64, device="cuda")
        for w in widths:
            sc, at = ((cum[w:] - cum[:-w]) / (sigma * math.sqrt(w))).max(0)
            up = sc > best
            best = torch.where(up, sc, best)
            bt[d] = torch.where(up, at.to(torch.int32), bt[d])
            bw[d] = torch.where(up, torch.full_like(bw[d], w), bw[d])
        snr[d] = best
    return {"dd": dd, "snr": snr, "t": bt, "w": bw, "n": (snr >= 6.0).sum().to(torch.int32).reshape(1)}


def _exact_gains(x, case):
    """The single-calibrator solution: from unit gains, E = mean_a g e conj(phi),
    g = phi sum_t E conj(e) / sum_t |e|^2, antenna 0's phase to 0, RMS |g| to 1; twice."""
    l, m = x["calibrator"]
    out = torch.empty((case["C"], case["A"], case["P"]), dtype=torch.complex128, device="cuda")
    for c in range(case["C"]):
        N = int(x["grid"][c])
        k = _cells(x["ant"], x["freq"][c], N)
        ph = torch.from_numpy(-2 * np.pi * 0.5 * (k[:, 0] * l + k[:, 1] * m)).cuda()
        phi = torch.polar(torch.ones_like(ph), ph)[:, None]
        e = _decode(x["v"][:, c])                                                # [T][A][P]
        den = (e.abs() ** 2).sum(0)
        g = torch.ones((case["A"], case["P"]), dtype=torch.complex128, device="cuda")
        for _ in range(2):
            E = (e * (g * phi.conj())[None]).mean(1)                             # [T][P]
            num = (E[:, None] * e.conj()).sum(0)
            g = torch.where(den > 0, phi * num / den.clamp(min=1), torch.zeros_like(num))
            g = g * (g[:1].conj() / g[:1].abs())
            g = g / (g.abs() ** 2).mean(0, keepdim=True).sqrt()
        out[c] = g
    return out


def exact(case, seed):
    if case["what"] == "search":
        return _exact_search(case, seed)
    x = _inputs(case, seed)
    T, C = case["T"], case["C"]
    if case["what"] == "gains":
        return _exact_gains(x, case)
    if case["what"] == "image":
        return torch.cat([_image(x, case, c, 0, T).reshape(-1) for c in range(C)])
    if case["what"] == "series":
        spi = case["spi"]
        return torch.stack([torch.cat([_image(x, case, c, t, t + spi).reshape(-1) for c in range(C)])
                            for t in range(0, T, spi)])
    return torch.cat([_fields(x, case, c, 0, T)[0].reshape(T, -1) for c in range(C)], dim=1)
