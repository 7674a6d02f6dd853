"""The work that is timed: calls a user of the library makes, through its public entry points.

Each case is a dict of plain values; `kind` says which call it is:

  search     Plan.search: a batch of DM-trial series to the ordered list of candidates
  spectrum   Plan.spectrum: real FFT and block-median normalisation of one series
  plane      Plan.power_plane: correlation of one spectrum with the template bank
  dedisperse DedispPlan.dedisperse: a filterbank to DM-trial series
  fourier    FourierPower forward and backward: P(r, z) and its gradient in the spectrum
  refine     Plan.refine: gradient ascent of candidate seeds

Inputs are N(0, 1) noise with weak accelerated sinusoids or pulse trains, as a
dedispersed survey series is after the observation's mean has been taken out;
filterbanks are N(0, 1) channels or 8-bit samples around 128.
"""
import math

import numpy as np
import torch

from paper_2211_13517_gb300 import capi

PREC = {"fp32": capi.FDAS_FP32, "bf16": capi.FDAS_BF16, "fp16": capi.FDAS_FP16}
DTYPE = {"fp32": torch.float32, "bf16": torch.bfloat16, "fp16": torch.float16}
TSAMP = 64e-6


def _search(name, n_log2, z_max, z_step, seg, harm, prec, series, **more):
    c = {"kind": "search", "n_log2": n_log2, "z_max": float(z_max), "z_step": float(z_step),
         "seg_len": seg, "n_harm": harm, "prec": prec, "series": series, "decimated": 0,
         "pulses": False, "host": False, "graph": False, "interbin": False, "fundamental": False,
         "sigma": 6.0}
    if name:
        c["name"] = name
    return {**c, **more}


def listed():
    return [
        # one short FP32 series with a coarse grid: an interactive look at one pointing, where
        # launches and host work count
        _search("search_short_fp32", 17, 16, 2, 2048, 4, "fp32", 1),
        # one full-length SKA-like series (600 s at 64 us) in plain FP32, with pulse trains
        _search("search_long_fp32", 23, 96, 1, 8192, 16, "fp32", 1, pulses=True),
        # a batch of such series with BF16 storage: the survey's production setting
        _search("search_batch_bf16", 23, 96, 1, 8192, 16, "bf16", 4),
        # an uneven batch out of page-locked host memory in FP16, replayed as a graph: high-DM
        # trials are decimated in time
        _search("search_uneven_fp16", 22, 96, 1, 8192, 16, "fp16", 6, decimated=6, host=True,
                graph=True),
        # a finer frequency grid on shorter series, eight harmonics
        _search("search_halfbin_bf16", 21, 50, 1, 4096, 8, "bf16", 2, interbin=True),
        # the correlation alone on the tensor cores: half-integer drift steps, an odd grid
        {"name": "plane_bf16", "kind": "plane", "n_log2": 21, "z_max": 45.0, "z_step": 0.5,
         "seg_len": 8192, "prec": "bf16"},
        # the same in FP32 with overlap-save transforms
        {"name": "plane_fp32", "kind": "plane", "n_log2": 20, "z_max": 96.0, "z_step": 2.0,
         "seg_len": 8192, "prec": "fp32"},
        # the spectrum of a full-length series with the block medians
        {"name": "spectrum_fp32", "kind": "spectrum", "n_log2": 23, "norm_block": 2048,
         "prec": "fp32"},
        # incoherent dedispersion: a small ragged FP32 filterbank
        {"name": "dedisperse_fp32", "kind": "dedisperse", "n_chan": 300, "n_out": (1 << 18) + 37,
         "n_dm": 75, "f_top": 1670.0, "df": 1.0, "dm_lo": 20.0, "dm_step": 0.1, "bits": 32},
        # and a survey's 8-bit one: 1024 channels, 128 trials
        {"name": "dedisperse_u8", "kind": "dedisperse", "n_chan": 1024, "n_out": 1 << 20,
         "n_dm": 128, "f_top": 1670.0, "df": 0.25, "dm_lo": 0.0, "dm_step": 0.25, "bits": 8},
        # differentiable Fourier-interpolated power at a few thousand points, gradient in the
        # spectrum (the one in (r, z) comes with the forward call)
        {"name": "fourier_power", "kind": "fourier", "n_log2": 20, "points": 3001, "z_abs": 90.0},
        # refinement of a search's candidates by gradient ascent
        {"name": "refine", "kind": "refine", "n_log2": 20, "points": 1024, "z_abs": 90.0,
         "steps": 50},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "plane", "plane", "spectrum", "dedisperse",
                       "dedisperse", "fourier", "refine"])
    if kind in ("search", "plane"):
        z_step = rng.choice([0.5, 1.0, 1.0, 2.0])
        z_max = z_step * rng.randint(0, min(96, int(96 / z_step)))
        seg = rng.choice([2048, 4096, 8192])
        prec = rng.choice(["fp32", "bf16", "bf16", "fp16"])
    if kind == "search":
        harm = rng.choice([1, 2, 4, 8, 8, 16, 16, 16, 32])
        n_log2 = rng.randint(12, 23)
        # at most the samples of four full-length series (two in FP32)
        top = max(1, min(24, (4 if prec != "fp32" else 1) << (23 - n_log2)))
        series = _log_int(rng, 1, top)
        dec = rng.choice([0, 0, series // 2]) if n_log2 >= 14 else 0
        host = rng.random() < 0.3
        n_z = 2 * round(z_max / z_step) + 1
        interbin = n_log2 <= 21 and n_z * series <= 800 and rng.random() < 0.25
        return _search(None, n_log2, z_max, z_step, seg, harm, prec, series, decimated=dec,
                       pulses=rng.random() < 0.3, host=host, graph=rng.random() < 0.3,
                       interbin=interbin, fundamental=rng.random() < 0.15,
                       sigma=round(rng.uniform(5.0, 8.0), 2))
    if kind == "plane":
        return {"kind": "plane", "n_log2": rng.randint(12, 22 if prec != "fp32" else 21),
                "z_max": z_max, "z_step": z_step, "seg_len": seg, "prec": prec}
    if kind == "spectrum":
        return {"kind": "spectrum", "n_log2": rng.randint(10, 24),
                "norm_block": rng.choice([256, 1024, 2048, 2048, 4096]),
                "prec": rng.choice(["fp32", "bf16", "fp16"])}
    if kind == "dedisperse":
        bits = rng.choice([8, 32])
        n_chan = _log_int(rng, 16, 1024)
        df = 256.0 / n_chan
        # additions bounded by the listed 8-bit filterbank's (a quarter of them in FP32)
        budget = (1 << 37) // (4 if bits == 32 else 1)
        n_dm = _log_int(rng, 1, 200)
        n_out = _log_int(rng, 1 << 12, max(1 << 13, min(1 << 20, budget // (n_chan * n_dm))))
        return {"kind": "dedisperse", "n_chan": n_chan, "n_out": n_out, "n_dm": n_dm,
                "f_top": 1670.0, "df": df, "dm_lo": round(rng.uniform(0.0, 100.0), 2),
                "dm_step": round(math.exp(rng.uniform(math.log(0.02), math.log(1.0))), 3),
                "bits": bits}
    points = _log_int(rng, 1, 8192 if kind == "fourier" else 1024)
    c = {"kind": kind, "n_log2": rng.randint(14, 21), "points": points,
         "z_abs": round(rng.uniform(0.0, 150.0), 1)}
    if kind == "refine":
        c["steps"] = rng.randint(1, 50)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _signals(seed, count, n, z_abs):
    """(r0, z0) of the injected signals, away from the ends of the spectrum."""
    r = np.random.RandomState(int(seed) % (1 << 31) + 17)
    return list(zip(r.uniform(0.02 * n, 0.45 * n, count), r.uniform(-z_abs, z_abs, count)))


def _series(n, seed, signals, pulses):
    """N(0, 1) samples with one weak accelerated signal per (r0, z0)."""
    x = torch.randn(n, generator=_generator(seed), device="cuda")
    if signals:
        u = torch.arange(n, device="cuda", dtype=torch.float64) / n
        for r0, z0 in signals:
            ph = r0 * u + z0 * (u - 0.5) ** 2 / 2.0
            if pulses:
                x += 0.054 * math.sqrt((1 << 23) / n) * ((ph - ph.floor()) < 0.05)
            else:
                amp = 0.05 * math.sqrt((1 << 17) / n)
                x += (amp * torch.cos(2.0 * math.pi * (ph - ph.floor()))).float()
    return x


def _n_z(case):
    return 2 * round(case["z_max"] / case["z_step"]) + 1


def _lengths(case):
    """The batch's lengths: the last `decimated` series shorter by 2, 4, 8 in turn."""
    n = 1 << case["n_log2"]
    full = case["series"] - case["decimated"] if case["decimated"] < case["series"] else case["series"]
    return [n] * full + [n >> (1 + i % 3) for i in range(case["decimated"])]


def _delays(case):
    """Delay table in samples [n_dm][n_chan], FP64 with one rounding per operation."""
    c = np.arange(case["n_chan"], dtype=np.float64)
    d = np.arange(case["n_dm"], dtype=np.float64)
    f = case["f_top"] - c * case["df"]
    a = 1.0 / (f * f) - 1.0 / (case["f_top"] * case["f_top"])
    dm = case["dm_lo"] + d * case["dm_step"]
    return np.floor(((4.148808e3 * dm)[:, None] * a[None, :]) / TSAMP + 0.5).astype(np.int64)


def prepare(case, seed):
    kind = case["kind"]
    n = 1 << case["n_log2"] if "n_log2" in case else 0
    if kind == "search":
        plan = capi.Plan(n, TSAMP, case["z_max"], case["z_step"], case["seg_len"], case["n_harm"],
                         precision=PREC[case["prec"]], threshold_sigma=case["sigma"],
                         use_graph=case["graph"], interbin=case["interbin"],
                         harmonic_mode=capi.FDAS_HARM_FUNDAMENTAL if case["fundamental"]
                         else capi.FDAS_HARM_TOP)
        xs = []
        for i, m in enumerate(_lengths(case)):
            s = 1000 * seed + i
            x = _series(m, s, _signals(s, 3 if case["pulses"] else 1, m, 0.9 * case["z_max"]),
                        case["pulses"])
            xs.append(x.cpu().pin_memory() if case["host"] else x)
        return {"kind": kind, "plan": plan, "series": xs,
                "stream": torch.cuda.Stream() if case["graph"] else None}
    if kind == "spectrum":
        plan = capi.Plan(n, TSAMP, 0.0, 1.0, 1024, 1, precision=PREC[case["prec"]],
                         norm_block=case["norm_block"])
        return {"kind": kind, "plan": plan, "x": _series(n, seed, _signals(seed, 1, n, 0.0), False)}
    if kind == "plane":
        plan = capi.Plan(n, TSAMP, case["z_max"], case["z_step"], case["seg_len"], 1,
                         precision=PREC[case["prec"]])
        return {"kind": kind, "plan": plan, "spec": _spectrum_input(case, seed)}
    if kind == "dedisperse":
        n_t = _n_t(case)
        dd = capi.DedispPlan(case["n_chan"], n_t, case["f_top"], case["df"], TSAMP, case["dm_lo"],
                             case["dm_step"], case["n_dm"], case["n_out"])
        return {"kind": kind, "plan": dd, "fb": _filterbank(case, seed)}
    plan = capi.Plan(n, TSAMP, 16.0, 2.0, 1024, 1)
    spec, rz = _points(case, seed)
    if kind == "fourier":
        g = torch.randn(case["points"], generator=_generator(seed + 5), device="cuda")
        return {"kind": kind, "plan": plan, "spec": spec.requires_grad_(True),
                "rz": torch.from_numpy(rz).cuda(), "g": g}
    seeds = np.zeros(case["points"], dtype=capi.SEED_DTYPE)
    seeds["r"], seeds["z"] = rz[:, 0], rz[:, 1]
    return {"kind": kind, "plan": plan, "spec": spec, "seeds": seeds, "steps": case["steps"]}


def _spectrum_input(case, seed):
    """A normalised spectrum: complex noise of unit mean power, 16 strong bins."""
    n_r = 1 << (case["n_log2"] - 1)
    x = torch.randn(2 * n_r, generator=_generator(seed), device="cuda") * math.sqrt(0.5)
    r = np.random.RandomState(int(seed) % (1 << 31))
    for k in r.randint(1, n_r, 16):
        x[2 * k] += 9.0
    x[:2] = 0.0
    return x.to(DTYPE[case["prec"]])


def _n_t(case):
    n_t = case["n_out"] + int(_delays(case)[-1, -1])
    return -(-n_t // 16) * 16


def _filterbank(case, seed):
    g = _generator(seed)
    shape = (case["n_chan"], _n_t(case))
    if case["bits"] == 32:
        return torch.randn(shape, generator=g, device="cuda")
    out = torch.empty(shape, dtype=torch.uint8, device="cuda")
    for c in range(0, shape[0], 64):
        y = torch.randn((min(64, shape[0] - c), shape[1]), generator=g, device="cuda")
        out[c:c + 64] = (y * 16.0 + 128.0).round_().clamp_(0, 255).to(torch.uint8)
    return out


def _points(case, seed):
    """A complex64 spectrum of unit noise power with 16 signals, and points near them: within
    half a bin and two units of drift, as the search's grid leaves them."""
    n = 1 << case["n_log2"]
    sig = _signals(seed, 16, n, case["z_abs"])
    x = _series(n, seed, sig, False)
    spec = (torch.fft.rfft(x.double())[:n // 2] / math.sqrt(n)).to(torch.complex64)
    spec[0] = 0
    r = np.random.RandomState(int(seed) % (1 << 31) + 3)
    which = r.randint(0, 16, case["points"])
    rz = np.array(sig)[which]
    rz[:, 0] += r.uniform(-0.5, 0.5, case["points"])
    rz[:, 1] += r.uniform(-2.0, 2.0, case["points"])
    return spec, rz


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    kind, plan = state["kind"], state["plan"]
    if kind == "search":
        out = np.zeros(1 << 14, dtype=capi.CANDIDATE_DTYPE)   # 0 past the last candidate
        status, _, n_found = plan.search(state["series"], stream=state["stream"], out=out)
        return {"status": status, "n_found": n_found, **{k: out[k] for k in out.dtype.names}}
    if kind == "spectrum":
        return plan.spectrum(state["x"], medians=True)
    if kind == "plane":
        return plan.power_plane(state["spec"])
    if kind == "dedisperse":
        return plan.dedisperse(state["fb"])
    if kind == "fourier":
        p = capi.FourierPower().apply(plan, state["spec"], state["rz"])
        (grad,) = torch.autograd.grad(p, state["spec"], state["g"])
        return {"power": p.detach(), "grad": grad}
    out = plan.refine(state["spec"], state["seeds"], n_steps=state["steps"])
    return {k: out[k].copy() for k in ("r", "z", "power", "dpdr", "dpdz", "steps")}


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------
def _correlation_flops(n_r, n_z, z_step):
    """The cheaper of the direct sums and of overlap-save transforms of 8192 points."""
    k = n_z // 2
    m = [8 + math.ceil(abs(i - k) * z_step / 2.0 - 1e-9) for i in range(n_z)]
    direct = 8.0 * n_r * sum(2 * mm + 1 for mm in m)
    seg = 8192.0
    fft = (5.0 * seg * math.log2(seg) + 9.0 * seg) * math.ceil(n_r / (seg - 2 * max(m))) * n_z
    return min(direct, fft)


def work(case):
    kind = case["kind"]
    size = 4 if case.get("prec") == "fp32" else 2
    if kind == "search":
        byts = flops = 0.0
        for n in _lengths(case):
            n_r = n // 2
            cells = _n_z(case) * n_r * (2 if case["interbin"] else 1)
            byts += 4.0 * n
            flops += 2.5 * n * math.log2(n) + _correlation_flops(n_r, _n_z(case), case["z_step"])
            flops += cells * (3.0 + case["n_harm"])
        return {"bytes": byts, "flops": flops}
    if kind == "spectrum":
        n = 1 << case["n_log2"]
        return {"bytes": 4.0 * n + size * n, "flops": 2.5 * n * math.log2(n) + 5.0 * n}
    if kind == "plane":
        n_r = 1 << (case["n_log2"] - 1)
        return {"bytes": 2.0 * size * n_r + float(size) * _n_z(case) * n_r,
                "flops": _correlation_flops(n_r, _n_z(case), case["z_step"])
                + 3.0 * _n_z(case) * n_r}
    if kind == "dedisperse":
        return {"bytes": case["n_chan"] * _n_t(case) * case["bits"] / 8.0
                + 4.0 * case["n_dm"] * case["n_out"],
                "flops": float(case["n_chan"]) * case["n_dm"] * case["n_out"]}
    # one evaluation: the window's sum at as many nodes as it has bins, with phases
    m = 32 + case["z_abs"] / 4.0
    one = 8.0 * (2 * m + 1) * 2 * m
    n_r = 1 << (case["n_log2"] - 1)
    if kind == "fourier":
        # forward, the forward sum again for the backward pass, and the window's responses
        return {"bytes": 8.0 * n_r + case["points"] * (16.0 + 4 + 4 + 16 * (2 * m + 1)),
                "flops": 3.0 * one * case["points"]}
    # the ascent stops early: about a third of the steps
    return {"bytes": case["points"] * (8.0 * (2 * m + 1) + 24 + 48),
            "flops": one * case["points"] * (1 + case["steps"] / 3.0)}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits, plain torch and numpy
# ---------------------------------------------------------------------------
def _nodes():
    u, w = np.polynomial.legendre.leggauss(640)
    return (torch.from_numpy(0.5 * (u + 1.0)).cuda(), torch.from_numpy(0.5 * w).cuda())


def _response(q, z):
    """rho(q, z) for the tensors q (any length) and the number z."""
    u, w = _nodes()
    ph = torch.outer(q - 0.5 * z, u) + 0.5 * z * u * u
    return torch.polar(torch.ones_like(ph), 2.0 * math.pi * ph) @ w.to(torch.complex128)


def exact(case, seed):
    kind = case["kind"]
    n_r = 1 << (case["n_log2"] - 1) if "n_log2" in case else 0
    if kind == "spectrum":
        n = 2 * n_r
        x = _series(n, seed, _signals(seed, 1, n, 0.0), False)
        X = torch.fft.rfft(x.double())[:n_r]
        X[0] = 0
        block = min(case["norm_block"], n_r)
        p = (X.real ** 2 + X.imag ** 2).reshape(-1, block)
        s = p.sort(dim=1).values
        med = 0.5 * (s[:, block // 2 - 1] + s[:, block // 2])
        med[0] = p[0, 1:].sort().values[(block - 1) // 2]
        X = X.reshape(-1, block) * torch.sqrt(math.log(2.0) / med)[:, None]
        return torch.view_as_real(X.reshape(-1)).reshape(-1), med
    if kind == "plane":
        if _n_z(case) * n_r > 3e8:
            return None
        X = torch.view_as_complex(_spectrum_input(case, seed).double().reshape(-1, 2))
        fx = torch.fft.fft(X, 2 * n_r)
        out = torch.empty((_n_z(case), n_r), dtype=torch.float64, device="cuda")
        for i in range(_n_z(case)):
            z = (i - _n_z(case) // 2) * case["z_step"]
            m = 8 + math.ceil(abs(z) / 2.0 - 1e-9)
            rho = _response(torch.arange(-m, m + 1, device="cuda", dtype=torch.float64), z)
            g = rho.conj() / torch.sqrt((rho.abs() ** 2).sum())
            f = torch.fft.ifft(fx * torch.fft.fft(g, 2 * n_r))[m:m + n_r]
            out[i] = f.real ** 2 + f.imag ** 2
        scale = 0.0625 if case["prec"] == "fp16" else 1.0
        return out * scale, torch.stack([out.mean(), out.std(unbiased=False)])
    if kind == "dedisperse":
        fb = _filterbank(case, seed)
        delays = _delays(case)
        out = torch.zeros((case["n_dm"], case["n_out"]), dtype=torch.float64, device="cuda")
        for c in range(case["n_chan"]):
            row = fb[c].double()
            for d in range(case["n_dm"]):
                k = int(delays[d, c])
                out[d] += row[k:k + case["n_out"]]
        return out
    if kind == "fourier":
        spec, rz = _points(case, seed)
        gp = torch.randn(case["points"], generator=_generator(seed + 5), device="cuda").double()
        X = spec.to(torch.complex128)
        u, w = _nodes()
        power = torch.empty(case["points"], dtype=torch.float64, device="cuda")
        grad = torch.zeros(n_r, dtype=torch.complex128, device="cuda")
        half = 32 + np.ceil(np.abs(rz[:, 1]) / 2.0 - 1e-12).astype(np.int64)
        half = np.minimum(half, 255)
        k0 = np.floor(rz[:, 0] + 0.5).astype(np.int64)
        for m in np.unique(half):
            at = np.nonzero(half == m)[0]
            e = torch.arange(-int(m), int(m) + 1, device="cuda")
            k = torch.from_numpy(k0[at]).cuda()[:, None] + e[None, :]
            inside = (k >= 0) & (k < n_r)
            k = k.clamp(0, n_r - 1)
            delta = torch.from_numpy(rz[at, 0] - k0[at]).cuda()
            z = torch.from_numpy(rz[at, 1]).cuda()
            th = (delta - 0.5 * z)[:, None] * u + 0.5 * z[:, None] * u * u
            A = torch.polar(torch.ones_like(th), 2.0 * math.pi * th) * w
            ph = torch.outer(u, e.double())
            rho = A @ torch.polar(torch.ones_like(ph), -2.0 * math.pi * ph)
            win = X[k] * inside
            F = (win * rho.conj()).sum(dim=1)
            i = torch.from_numpy(at).cuda()
            power[i] = F.real ** 2 + F.imag ** 2
            add = (2.0 * gp[i] * F)[:, None] * rho * inside
            grad.index_add_(0, k.reshape(-1), add.reshape(-1))
        return {"power": power, "grad": grad}
    # a search's list and an ascent's end follow from comparisons of rounded values
    return None
