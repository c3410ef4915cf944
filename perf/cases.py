"""Workloads of the F-statistic library, one pass of each through its public
entry points, with an FP64 statement of what the pass returns.

``listed()`` names the workloads a search runs; ``draw(rng)`` gives further
ones of the same ranges.  ``prepare`` makes what a program holds before the
call (series, templates, gaps, plan), ``run`` is one call of the program,
``work`` the bytes and operations the call cannot do without, ``exact`` its
results in 64 bits by plain torch.
"""
from __future__ import annotations

import dataclasses
import math
import random

import numpy as np
import torch

import paper_0912_4255_gb300 as fs
from paper_0912_4255_gb300.autograd import BinSearch, FStatBin
from paper_0912_4255_gb300.batch import RaggedBatch

DEV = "cuda"
C_LIGHT = 299792458.0
HOUR = 3600.0


# ------------------------------------------------------------------ plan data
@dataclasses.dataclass
class Site:
    lat_rad: float = math.radians(46.45)
    lon_rad: float = math.radians(-119.41)
    gamma_rad: float = math.radians(171.8)
    radius_m: float = 6371000.0


@dataclasses.dataclass
class Orbit:
    au_m: float = 1.495978707e11
    year_s: float = 365.25 * 86400.0
    sidereal_day_s: float = 86164.0905
    obliquity_rad: float = math.radians(23.44)
    orb_phase0: float = 0.0
    sid_phase0: float = 0.0


@dataclasses.dataclass
class Desc:
    dt: float = 0.5
    t_start: float = 0.0
    n_data: int = 86400
    f_het: float = 100.0
    sigma2: float = 1.0
    n_fft: int = 1 << 17
    interp: int = fs.SINC
    taps: int = 8
    window: int = fs.WIN_LANCZOS
    precision: int = fs.PREC_MIXED
    det: Site = dataclasses.field(default_factory=Site)
    eph: Orbit = dataclasses.field(default_factory=Orbit)
    max_templates: int = 1

    def replace(self, **kw):
        return dataclasses.replace(self, **kw)


@dataclasses.dataclass
class SftDesc:
    sft_len: int
    dt_raw: float
    k_lo: int
    n_bins: int
    k_het: int
    band_bins: int
    dirichlet_terms: int = 16
    median_window: int = 101
    tukey_frac: float = 0.05
    edge_taper: int = 0


def pow2(n):
    return 1 << max(12, int(n - 1).bit_length())


def compute_case(name, n_data, n_t, n_fft=0, dt=0.5, f_het=100.0, taps=8, window="lanczos", precision="mixed",
                 gap_frac=0.1, fdot_min=-1e-9, half_band=False, entry="plan"):
    """taps = 0: nearest neighbour.  entry: "plan" (fstat_compute) or
    "noalloc" (fstat_compute_noalloc)."""
    c = dict(kind="compute", n_data=n_data, n_t=n_t, n_fft=n_fft or pow2(int(n_data * 1.0002) + 3), dt=dt, f_het=f_het,
             taps=taps, window=window, precision=precision, gap_frac=gap_frac, fdot_min=fdot_min,
             half_band=half_band, entry=entry)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one sky position, 12 h at 2 Hz, nearest neighbour (the quick look and the smoke run)
        compute_case("one_12h_nearest", 86400, 1, 1 << 17, taps=0, gap_frac=0.0),
        # one template of a 10 d search, as a candidate is looked at again
        compute_case("one_10d_sinc8", 1_728_000, 1, 1 << 22),
        # the search itself: 10 d, 10 % gaps, one chunk of its sky x spindown grid
        compute_case("search_10d_sinc8", 1_728_000, 64, 1 << 22),
        # band doubling: 5.3 d at 4 Hz, plain truncated sinc, the central half of the band kept; an odd length
        compute_case("doubled_band_5d", 1_831_681, 12, dt=0.25, window="rect", half_band=True),
        # 30 d at 1 kHz, the longest FFT and the fastest phase
        compute_case("long_30d_1khz", 10_368_000, 2, 1 << 24, dt=0.25, f_het=1000.0, gap_frac=0.0, fdot_min=-1e-8),
        # the all-FP64 mode that a result is checked with
        compute_case("one_10d_fp64", 1_728_000, 1, 1 << 22, precision="fp64"),
        # a search over uneven spans, each template with its own gaps, one CUDA graph
        dict(name="ragged_1_to_10d", kind="ragged", n_t=48, n_data=1_728_000, min_days=1.0, max_days=10.0),
        # Monte Carlo: noise, one signal per 12 h realization, 2F of each
        dict(name="monte_carlo_12h", kind="montecarlo", realizations=128, span=86400),
        # follow-up of candidates by gradient ascent: 2F and its gradient
        dict(name="gradient_5d", kind="grad", n_t=64, n_data=864_000, gap_frac=0.1, taps=8),
        # the loudest bins of every band of a block of 2F spectra
        dict(name="candidates_16_rows", kind="topk", n_rows=16, row_len=1 << 22, band_len=65536, k=16),
        # 10 d of 1800 s SFTs to the heterodyned series of the search
        dict(name="front_end_10d", kind="sft", slots=480, missing=48, t_sft=1800.0, band_bins=3600, dk=16, median=101),
        # the earlier method on the same SFTs
        dict(name="sft_demod_10d", kind="demod", slots=480, missing=48, t_sft=1800.0, band_bins=3600, dk=16, n_t=4,
             n_q=32768),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["compute", "compute", "compute", "compute", "ragged", "montecarlo", "grad", "topk", "sft",
                       "demod", "inject"])
    if kind == "compute":
        n_data = _spread(rng, 20_000, 4_000_000) | 1
        n_fft = pow2(int(n_data * 1.0002) + 3) * rng.choice([1, 1, 2])
        precision = rng.choice(["mixed", "mixed", "mixed", "mixed", "fp64"])
        n_t = min(_spread(rng, 1, 64), max(1, (1 << (27 if precision == "mixed" else 22)) // n_fft))
        taps = rng.choice([0, 8, 8, 8, 4, 16])
        entry = "noalloc" if precision == "mixed" and n_fft <= 1 << 20 and rng.random() < 0.2 else "plan"
        return compute_case("", n_data, min(n_t, 6) if entry == "noalloc" else n_t, n_fft,
                            dt=rng.choice([0.25, 0.5, 0.5, 1.0]), f_het=rng.choice([50.0, 100.0, 100.0, 1000.0]),
                            taps=taps, window=rng.choice(["lanczos", "lanczos", "rect"]), precision=precision,
                            gap_frac=rng.choice([0.0, 0.05, 0.1, 0.2]), half_band=rng.random() < 0.25 and entry == "plan",
                            entry=entry)
    if kind == "ragged":
        hi = rng.uniform(2.0, 10.0)
        return dict(kind=kind, n_t=_spread(rng, 4, 48), n_data=1_728_000, min_days=1.0, max_days=hi)
    if kind == "montecarlo":
        return dict(kind=kind, realizations=_spread(rng, 4, 128), span=86400 - rng.randrange(0, 40000))
    if kind == "grad":
        return dict(kind=kind, n_t=_spread(rng, 1, 64), n_data=_spread(rng, 60_000, 860_000) | 1, gap_frac=rng.choice([0.0, 0.1, 0.2]),
                    taps=rng.choice([8, 8, 8, 4, 16]))
    if kind == "topk":
        band_len = 2048 << rng.randrange(0, 8)
        row_len = band_len * rng.randrange(1, max(2, (1 << 22) // band_len))
        return dict(kind=kind, n_rows=rng.randrange(1, 17), row_len=row_len, band_len=band_len, k=rng.choice([1, 4, 16, 16, 64]))
    if kind in ("sft", "demod"):
        slots = _spread(rng, 20, 480)
        c = dict(kind=kind, slots=slots, missing=int(slots * rng.choice([0.0, 0.1, 0.2])), t_sft=1800.0,
                 band_bins=rng.choice([900, 1800, 2400, 3600]), dk=rng.choice([8, 16, 16]))
        if kind == "sft":
            return dict(c, median=rng.choice([51, 101, 101]))
        return dict(c, n_t=rng.randrange(1, 5), n_q=_spread(rng, 1000, 32768))
    return dict(kind="inject", n_inj=_spread(rng, 1, 256), span=_spread(rng, 20_000, 200_000) | 1)


# ------------------------------------------------------------------ inputs
def _np(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _noise(n, seed):
    return (torch.randn(2 * n, generator=_gen(seed), device=DEV) * math.sqrt(0.5)).view(torch.complex64)


def _gaps(n, frac, dt, seed, lo=0):
    """Sorted, disjoint [start, end) blocks of 1-6 h covering about frac of n samples."""
    g = _np(seed)
    hour = max(2, int(HOUR / dt))
    iv, covered, tries = [], 0, 0
    while covered < frac * n and tries < 2000:
        tries += 1
        ln = int(g.integers(hour, 6 * hour + 1))
        if ln >= n // 3:
            ln = max(1, n // 8)
        s = int(g.integers(1, n - ln - 1))
        if all(s + ln + 1 <= a or s >= b + 1 for a, b in iv):
            iv.append((s, s + ln))
            covered += ln
    iv.sort()
    return np.asarray(iv, np.int64).reshape(-1, 2) + lo


def _templates(n, seed, span_start, span_len, fdot_min=-1e-9):
    g = _np(seed)
    t = np.zeros(n, fs.TEMPLATE_DTYPE)
    t["alpha"] = g.uniform(0, 2 * math.pi, n)
    t["delta"] = np.arcsin(g.uniform(-1, 1, n))
    t["fdot"] = g.uniform(fdot_min, 0.0, n)
    t["span_start"] = span_start
    t["span_len"] = span_len
    t["out_off"] = -1
    return t


def _injections(n, seed, span_start, span_len, df):
    g = _np(seed)
    r = np.zeros(n, fs.INJECTION_DTYPE)
    r["alpha"] = g.uniform(0, 2 * math.pi, n)
    r["delta"] = np.arcsin(g.uniform(-1, 1, n))
    r["psi"] = g.uniform(0, math.pi, n)
    r["cosi"] = g.uniform(-1, 1, n)
    r["phi0"] = g.uniform(0, 2 * math.pi, n)
    r["h0"] = 0.12
    r["df"] = df
    r["span_start"] = span_start
    r["span_len"] = span_len
    return r


def _desc(c):
    return Desc(dt=c["dt"], n_data=c["n_data"], f_het=c["f_het"], n_fft=c["n_fft"],
                interp=fs.SINC if c["taps"] else fs.NEAREST, taps=c["taps"] or 8,
                window=fs.WIN_LANCZOS if c["window"] == "lanczos" else fs.WIN_RECT,
                precision=fs.PREC_FP64 if c["precision"] == "fp64" else fs.PREC_MIXED, max_templates=c["n_t"])


def _compute_inputs(c, seed):
    d = _desc(c)
    x = _noise(d.n_data, seed)
    gaps = _gaps(d.n_data, c["gap_frac"], d.dt, seed + 1)
    for a, b in gaps:
        x[a:b] = 0
    t = _templates(c["n_t"], seed + 2, 0, d.n_data, c["fdot_min"])
    t["n_gaps"] = len(gaps)
    return d, x, t, gaps


def _ragged_inputs(c, seed):
    d = Desc(n_data=c["n_data"], n_fft=1 << 21, max_templates=c["n_t"])
    g = _np(seed)
    day = int(86400 / d.dt)
    x = _noise(d.n_data, seed)
    n = c["n_t"]
    # spans evenly spread over the range, in a scattered order (the same for every seed: so is the output's length)
    frac = ((np.arange(n) * 0.6180339887498949) % 1.0)
    lens = np.minimum(((c["min_days"] + frac * (c["max_days"] - c["min_days"])) * day).astype(np.int64), d.n_data)
    starts = np.array([int(g.integers(0, d.n_data - L + 1)) for L in lens])
    t = _templates(n, seed + 2, starts, lens)
    lists, off, pos = [], 0, 0
    for i in range(n):
        gi = _gaps(int(lens[i]), float(g.uniform(0, 0.2)), d.dt, seed * 1000 + i, int(starts[i]))
        nf = pow2(int(lens[i] * 1.0002) + 3)
        t["gap_off"][i], t["n_gaps"][i], t["n_fft"][i], t["out_off"][i] = off, len(gi), nf, pos
        lists.append(gi)
        off += len(gi)
        pos += nf
    return d, x, t, np.concatenate(lists)


def _mc_inputs(c, seed):
    r, span = c["realizations"], c["span"]
    d = Desc(n_data=r * span, n_fft=pow2(int(span * 1.0002) + 3), interp=fs.NEAREST, max_templates=r)
    starts = np.arange(r) * span
    inj = _injections(r, seed + 3, starts, span, 3000 / (d.n_fft * d.dt))
    t = _templates(r, seed + 2, starts, span, 0.0)
    t["alpha"], t["delta"] = inj["alpha"], inj["delta"]
    return d, _noise(d.n_data, seed), inj, t


def _grad_inputs(c, seed):
    n, n_t = c["n_data"], c["n_t"]
    d = Desc(n_data=n, n_fft=pow2(int(n * 1.0002) + 3), taps=c["taps"], max_templates=n_t)
    g = _np(seed)
    gaps = _gaps(n, c["gap_frac"], d.dt, seed + 1)
    T = n * d.dt
    inj = _injections(min(20, n_t), seed + 3, 0, n, 0.0)
    inj["df"] = g.uniform(0.05, 0.4, len(inj))
    inj["fdot"] = g.uniform(-1e-9, 0, len(inj))
    inj["h0"] = 60.0 / math.sqrt(n)
    x = _noise(n, seed).to(torch.complex128)
    for i in inj:
        x += _signal(i, d)
    x = x.to(torch.complex64)
    for a, b in gaps:
        x[a:b] = 0
    src = np.arange(n_t) % len(inj)
    theta = np.stack([inj["alpha"][src] + g.uniform(-3e-4, 3e-4, n_t), inj["delta"][src] + g.uniform(-3e-4, 3e-4, n_t),
                      inj["df"][src] + g.uniform(-0.3, 0.3, n_t) / T, inj["fdot"][src] + g.uniform(-0.3, 0.3, n_t) / T ** 2], 1)
    t = _templates(n_t, seed + 2, 0, n)
    t["alpha"], t["delta"], t["fdot"] = theta[:, 0], theta[:, 1], theta[:, 3]
    t["n_gaps"] = len(gaps)
    return d, x, t, gaps, torch.from_numpy(theta).to(DEV)


def _topk_input(c, seed):
    # 2F of noise: chi-squared with four degrees of freedom
    z = torch.rand(2, c["n_rows"] * c["row_len"], generator=_gen(seed), device=DEV).clamp_min_(1e-12)
    return -2.0 * (z[0].log() + z[1].log())


def _sft_inputs(c, seed):
    n1, dk, pad, fs_raw = c["band_bins"], c["dk"], 8, 256.0
    k_h = int(100.0 * c["t_sft"])
    d = SftDesc(int(c["t_sft"] * fs_raw), 1.0 / fs_raw, k_h - n1 // 2 - dk - pad, n1 + 2 * (dk + pad), k_h, n1, dk,
                c.get("median", 101))
    g = _np(seed)
    keep = np.ones(c["slots"], bool)
    while (~keep).sum() < c["missing"]:
        a = int(g.integers(1, c["slots"]))
        keep[a:a + int(g.integers(1, 4))] = False
    slots = np.nonzero(keep)[0]
    X = (_noise(len(slots) * d.n_bins, seed) * math.sqrt(d.sft_len)).view(len(slots), d.n_bins)
    return d, X, slots * c["t_sft"]


def _demod_inputs(c, seed):
    d, X, t = _sft_inputs(c, seed)
    n = c["slots"] * c["band_bins"]
    dt = c["t_sft"] / c["band_bins"]
    plan = Desc(dt=dt, n_data=n, n_fft=pow2(n) * 2, f_het=d.k_het / c["t_sft"], max_templates=c["n_t"])
    return d, X / math.sqrt(d.sft_len), t, plan, _templates(c["n_t"], seed + 2, 0, n)


def _gap_tensor(gaps):
    return torch.from_numpy(np.ascontiguousarray(gaps).reshape(-1)).to(DEV)


# ------------------------------------------------------------------ one pass
def prepare(case, seed):
    k = case["kind"]
    s = dict(case=case)
    if k == "compute":
        d, x, t, gaps = _compute_inputs(case, seed)
        s.update(desc=d, x=x, t=fs.pack_templates(t, device=DEV), gaps=_gap_tensor(gaps))
        if case["entry"] == "plan":
            s["plan"] = fs.Plan(d, device=DEV)
            if case["half_band"]:
                s["plan"].keep_lower_half()
            s["out"] = torch.empty(case["n_t"] * s["plan"].band_len(), device=DEV)
        else:
            s["out"] = torch.empty(case["n_t"] * d.n_fft, device=DEV)
    elif k == "ragged":
        d, x, t, gaps = _ragged_inputs(case, seed)
        torch.cuda.synchronize()
        s["batch"] = RaggedBatch(d, x, t, _gap_tensor(gaps), device=DEV, graph=True)
    elif k == "montecarlo":
        d, x, inj, t = _mc_inputs(case, seed)
        rec, longest = fs.pack_injections(inj, device=DEV)
        s.update(plan=fs.Plan(d, device=DEV), noise=x, x=torch.empty_like(x), inj=rec, longest=longest,
                 t=fs.pack_templates(t, device=DEV), out=torch.empty(case["realizations"] * d.n_fft, device=DEV))
    elif k == "grad":
        d, x, t, gaps, theta = _grad_inputs(case, seed)
        s.update(search=BinSearch(fs.Plan(d, device=DEV), x, t, _gap_tensor(gaps)), theta=theta.requires_grad_())
    elif k == "topk":
        nb = case["row_len"] // case["band_len"]
        s.update(f=_topk_input(case, seed), val=torch.empty(case["n_rows"], nb, case["k"], device=DEV),
                 bins=torch.empty(case["n_rows"], nb, case["k"], dtype=torch.int32, device=DEV))
    elif k == "sft":
        d, X, t = _sft_inputs(case, seed)
        n = case["slots"] * case["band_bins"]
        s.update(d=d, X=X, t=t, n=n, x=torch.empty(n, dtype=torch.complex64, device=DEV),
                 ws=torch.empty(fs.fstat_sft_workspace(d, len(t)) + 256, dtype=torch.uint8, device=DEV))
    elif k == "demod":
        d, X, t, pd, tm = _demod_inputs(case, seed)
        plan = fs.Plan(pd, device=DEV)
        s.update(d=d, X=X, ts=torch.from_numpy(t).to(DEV), plan=plan, t=fs.pack_templates(tm, device=DEV),
                 out=torch.empty(case["n_t"], case["n_q"], device=DEV), q0=pd.n_fft // 2 - case["n_q"] // 2,
                 ws=torch.empty(int(plan.lib.fstat_sft_demod_workspace(len(t), case["n_t"])) + 256, dtype=torch.uint8,
                                device=DEV))
    else:
        span, n = case["span"], case["n_inj"] * case["span"]
        d = Desc(n_data=n, interp=fs.NEAREST, n_fft=pow2(int(span * 1.0002) + 3))
        rec, longest = fs.pack_injections(_injections(case["n_inj"], seed + 3, np.arange(case["n_inj"]) * span, span, 0.02),
                                          device=DEV)
        s.update(plan=fs.Plan(d, device=DEV), inj=rec, longest=longest, x=torch.empty(n, dtype=torch.complex64, device=DEV))
    return s


def run(s):
    c = s["case"]
    k = c["kind"]
    if k == "compute":
        if c["entry"] == "plan":
            return fs.fstat_compute(s["plan"], s["x"], s["t"], s["gaps"], s["out"])
        return fs.fstat_compute_noalloc(s["desc"], s["x"], s["t"], s["gaps"], s["out"])
    if k == "ragged":
        b = s["batch"]
        b.stream.wait_stream(torch.cuda.current_stream())
        out = b.run()
        torch.cuda.current_stream().wait_stream(b.stream)
        return out
    if k == "montecarlo":
        s["x"].copy_(s["noise"])
        fs.fstat_inject(s["plan"], s["x"], s["inj"], s["longest"])
        return {"x": s["x"], "two_f": fs.fstat_compute(s["plan"], s["x"], s["t"], None, s["out"])}
    if k == "grad":
        two_f = FStatBin.apply(s["theta"], s["search"])
        (g,) = torch.autograd.grad(two_f.sum(), s["theta"])
        # a mixed-precision plan evaluates in FP32: the candidate table keeps float32, as every 2F of the library
        return {"two_f": two_f.detach().float(), "grad": g.float()}
    if k == "topk":
        return fs.fstat_topk(s["f"], c["band_len"], c["k"], c["n_rows"], val=s["val"], bins=s["bins"])
    if k == "sft":
        return fs.fstat_sft_series(s["d"], s["X"], s["t"], 0.0, s["n"], x_h=s["x"], workspace=s["ws"])
    if k == "demod":
        return fs.fstat_sft_demod(s["plan"], s["d"], s["X"], s["ts"], s["t"], s["q0"], c["n_q"], twoF=s["out"],
                                  workspace=s["ws"])
    s["x"].zero_()
    return fs.fstat_inject(s["plan"], s["x"], s["inj"], s["longest"])


def work(case):
    """Inputs read once, outputs written once; operations of the resampler
    (taps x (weight, complex MAC) + time map, rotation, weights), of two FFTs
    and of 2F."""
    k = case["kind"]

    def search(n_data, n_fft, n_t, taps, out):
        per = n_data * (9 * max(taps, 1) + 16) + 2 * 5 * n_fft * math.log2(n_fft) + 12 * n_fft
        return {"bytes": 8.0 * n_data + 4.0 * out * n_t, "flops": per * n_t}

    if k == "compute":
        return search(case["n_data"], case["n_fft"], case["n_t"], case["taps"],
                      case["n_fft"] // 2 if case["half_band"] else case["n_fft"])
    if k == "ragged":
        n = (case["min_days"] + case["max_days"]) / 2 * 172800.0
        w = search(n, 1.5 * n, case["n_t"], 8, 1.5 * n)
        return dict(w, bytes=w["bytes"] + 8.0 * (case["n_data"] - n))
    if k == "montecarlo":
        span, r = case["span"], case["realizations"]
        n = pow2(int(span * 1.0002) + 3)
        w = search(span, n, r, 0, n)
        return {"bytes": 16.0 * span * r + 4.0 * n * r, "flops": w["flops"] + 60.0 * span * r}
    if k == "grad":
        return {"bytes": 8.0 * case["n_data"] + 112.0 * case["n_t"],
                "flops": case["n_t"] * case["n_data"] * (9.0 * case["taps"] + 40 + 14.0 * case["taps"] + 120)}
    if k == "topk":
        n = case["n_rows"] * case["row_len"]
        return {"bytes": 4.0 * n + 8.0 * case["n_rows"] * (case["row_len"] // case["band_len"]) * case["k"], "flops": 1.0 * n}
    n_sft = case.get("slots", 0) - case.get("missing", 0)
    if k == "sft":
        n1 = case["band_bins"]
        bins = n_sft * (n1 + 2 * case["dk"] + 16)
        return {"bytes": 8.0 * bins + 8.0 * n1 * case["slots"],
                "flops": n_sft * n1 * (4.0 * (2 * case["dk"] + 1) + 2 * 5 * math.log2(max(2, n1 * n_sft)))}
    if k == "demod":
        return {"bytes": 8.0 * n_sft * (case["band_bins"] + 2 * case["dk"] + 16) + 4.0 * case["n_t"] * case["n_q"],
                "flops": case["n_t"] * case["n_q"] * n_sft * (6.0 * (2 * case["dk"] + 1) + 40)}
    return {"bytes": 8.0 * case["n_inj"] * case["span"], "flops": 60.0 * case["n_inj"] * case["span"]}


# ------------------------------------------------------------------ in 64 bits
TAU = 2 * math.pi


def _f64(v):
    return torch.as_tensor(v, dtype=torch.float64, device=DEV)


def _hour(t, alpha, d):
    return d.eph.sid_phase0 + d.det.lon_rad + TAU * t / d.eph.sidereal_day_s - alpha


def _delay(t, alpha, delta, d):
    """Roemer delay n . r_d / c (s)."""
    e = d.eph
    ca, sa, cd, sd = torch.cos(alpha), torch.sin(alpha), torch.cos(delta), torch.sin(delta)
    phi = e.orb_phase0 + TAU * t / e.year_s
    ce, se = math.cos(e.obliquity_rad), math.sin(e.obliquity_rad)
    cl, sl = math.cos(d.det.lat_rad), math.sin(d.det.lat_rad)
    au, r = e.au_m / C_LIGHT, d.det.radius_m / C_LIGHT
    return (au * (cd * ca * torch.cos(phi) + (ce * cd * sa + se * sd) * torch.sin(phi))
            + r * (cl * cd * torch.cos(_hour(t, alpha, d)) + sl * sd))


def _rate(t, alpha, delta, d):
    e = d.eph
    ca, sa, cd, sd = torch.cos(alpha), torch.sin(alpha), torch.cos(delta), torch.sin(delta)
    wo, ws = TAU / e.year_s, TAU / e.sidereal_day_s
    phi = e.orb_phase0 + wo * t
    ce, se = math.cos(e.obliquity_rad), math.sin(e.obliquity_rad)
    au, r = e.au_m / C_LIGHT, d.det.radius_m / C_LIGHT
    return (au * wo * (-cd * ca * torch.sin(phi) + (ce * cd * sa + se * sd) * torch.cos(phi))
            - r * ws * math.cos(d.det.lat_rad) * cd * torch.sin(_hour(t, alpha, d)))


def _beams(t, alpha, delta, d):
    """Jaranowski-Krolak-Schutz a(t), b(t), arms at 90 degrees."""
    lam, gam = d.det.lat_rad, d.det.gamma_rad
    s2g, c2g, sl, cl = math.sin(2 * gam), math.cos(2 * gam), math.sin(lam), math.cos(lam)
    c2l, s2l = math.cos(2 * lam), math.sin(2 * lam)
    sd, cd, s2d, c2d = torch.sin(delta), torch.cos(delta), torch.sin(2 * delta), torch.cos(2 * delta)
    x = -_hour(t, alpha, d)
    a = (s2g * (3 - c2l) * (3 - c2d) * torch.cos(2 * x) / 16 - c2g * sl * (3 - c2d) * torch.sin(2 * x) / 4
         + s2g * s2l * s2d * torch.cos(x) / 4 - c2g * cl * s2d * torch.sin(x) / 2 + 0.75 * s2g * cl * cl * cd * cd)
    b = (c2g * sl * sd * torch.cos(2 * x) + s2g * (3 - c2l) * sd * torch.sin(2 * x) / 4 + c2g * cl * cd * torch.cos(x)
         + s2g * s2l * cd * torch.sin(x) / 2)
    return a, b


def _cis(cycles):
    r = (cycles - torch.round(cycles)) * TAU
    return torch.complex(torch.cos(r), torch.sin(r))


def _series(x, valid, tmpl, d, theta=None):
    """Weighted series of one template: (y a, y b, mask, a, b, tau_b); theta
    (alpha, delta, f, fdot) as differentiable scalars, else the record's."""
    alpha, delta, fdot = (theta[0], theta[1], theta[3]) if theta is not None else (
        _f64(float(tmpl["alpha"])), _f64(float(tmpl["delta"])), _f64(float(tmpl["fdot"])))
    lo = int(tmpl["span_start"])
    ends = _f64([d.t_start + lo * d.dt, d.t_start + (lo + int(tmpl["span_len"]) - 1) * d.dt])
    tb_ends = ends + _delay(ends, alpha, delta, d)
    with torch.no_grad():
        n_b = int(torch.floor((tb_ends[1] - tb_ends[0]) / d.dt)) + 1
    tb = tb_ends[0] + torch.arange(n_b, dtype=torch.float64, device=DEV) * d.dt
    with torch.no_grad():
        T = tb - _delay(tb, alpha, delta, d)
        for _ in range(5):
            T = tb - _delay(T, alpha, delta, d)
        r = 1 + _rate(T, alpha, delta, d)
    T = T - (T + _delay(T, alpha, delta, d) - tb) / r
    u = (T - d.t_start) / d.dt
    n = x.numel()
    with torch.no_grad():
        near = torch.floor(u + 0.5).long()
        inside = (near >= 0) & (near < n)
        m = (valid[near.clamp(0, n - 1)] & inside).double()
        base = torch.floor(u).long()
    if d.interp == fs.NEAREST:
        z = torch.where(inside, x[near.clamp(0, n - 1)], 0)
    else:
        half = d.taps // 2
        z = 0
        for i in range(d.taps):
            j = base - half + 1 + i
            jc = j.clamp(0, n - 1)
            v = torch.where((j >= 0) & (j < n) & valid[jc], x[jc], 0)
            w = torch.sinc(u - j)
            if d.window == fs.WIN_LANCZOS:
                w = w * torch.sinc((u - j) / half)
            z = z + v * w
    tau_b = tb - d.t_start
    a, b = _beams(T, alpha, delta, d)
    fdd = float(tmpl["fddot"])
    y = m * z * _cis(-(d.f_het * _delay(T, alpha, delta, d) + 0.5 * fdot * tau_b ** 2 + fdd * tau_b ** 3 / 6))
    return a * y, b * y, m, a, b, tau_b


def _two_f(Fa, Fb, m, a, b, sigma2):
    A, B, C = (m * a * a).sum(), (m * b * b).sum(), (m * a * b).sum()
    q = B * (Fa * Fa.conj()).real + A * (Fb * Fb.conj()).real - 2 * C * (Fa * Fb.conj()).real
    return 2 * q / (sigma2 * (A * B - C * C))


def _valid(d, tmpl, gaps):
    v = torch.zeros(d.n_data, dtype=torch.bool, device=DEV)
    lo = int(tmpl["span_start"])
    v[lo:lo + int(tmpl["span_len"])] = True
    for s, e in gaps[int(tmpl["gap_off"]):int(tmpl["gap_off"]) + int(tmpl["n_gaps"])]:
        v[int(s):int(e)] = False
    return v


def _spectrum(x, tmpl, gaps, d, n_fft, band=None):
    wa, wb, m, a, b, _ = _series(x, _valid(d, tmpl, gaps), tmpl, d)
    Fa, Fb = (torch.fft.fftshift(torch.fft.fft(w, n=n_fft)) for w in (wa, wb))
    f = _two_f(Fa, Fb, m, a, b, d.sigma2)
    return f if band is None else f[band[0]:band[1]]


def _signal(i, d):
    """Heterodyned positive-frequency half of one injection over its span."""
    n = int(i["span_start"]) + torch.arange(int(i["span_len"]), dtype=torch.float64, device=DEV)
    t = d.t_start + n * d.dt
    al, de = _f64(float(i["alpha"])), _f64(float(i["delta"]))
    tm = _delay(t, al, de, d)
    tau = n * d.dt + tm
    a, b = _beams(t, al, de, d)
    c2, s2 = math.cos(2 * i["psi"]), math.sin(2 * i["psi"])
    Ap, Ax = i["h0"] * (1 + i["cosi"] ** 2) / 2, i["h0"] * i["cosi"]
    cyc = (d.f_het * tm + float(i["df"]) * tau + 0.5 * float(i["fdot"]) * tau ** 2 + float(i["fddot"]) * tau ** 3 / 6
           + i["phi0"] / TAU)
    amp = torch.complex((a * c2 + b * s2) * Ap, -(b * c2 - a * s2) * Ax)
    return 0.5 * amp * _cis(cyc)


def _normalised(X, w):
    P = X.abs() ** 2
    K, h = P.shape[1], w // 2
    S = torch.empty_like(P)
    for k in range(K):
        win = P[:, max(0, k - h):min(K, k + h + 1)].sort(dim=1).values
        S[:, k] = win[:, (win.shape[1] - 1) // 2]
    return X / torch.sqrt(S / math.log(2.0))


def _sft_series_exact(d, X, t, n):
    X = _normalised(X.to(torch.complex128), d.median_window)
    t_len = d.sft_len * d.dt_raw
    n1, dk = d.band_bins, d.dirichlet_terms
    out = torch.zeros(n, dtype=torch.complex128, device=DEV)
    a = 0
    for i in range(1, len(t) + 1):
        if i < len(t) and abs(t[i] - t[i - 1] - t_len) <= 1e-6 * t_len:
            continue
        M = i - a
        D = torch.fft.fft(X[a:i], dim=0)                      # sum over the SFTs of the chunk, per r
        r = torch.arange(M, dtype=torch.float64, device=DEV)[:, None]
        k0 = d.k_het - n1 // 2 - d.k_lo
        Xb = torch.zeros(M, n1, dtype=torch.complex128, device=DEV)
        for j in range(-dk, dk + 1):
            y = TAU * (r / M - j)
            ys = torch.where(y == 0, 1.0, y)
            P = torch.complex(torch.where(y == 0, 1.0, torch.sin(y) / ys), torch.where(y == 0, 0.0, -(1 - torch.cos(y)) / ys))
            Xb += D[:, k0 + j:k0 + j + n1] * P
        spec = Xb.T.reshape(-1)                               # m = kappa M + r, ascending
        no = n1 * M
        xx = (torch.arange(no, dtype=torch.float64, device=DEV) + 0.5) / no
        e = d.tukey_frac / 2
        w = torch.ones_like(xx)
        w = torch.where(xx < e, 0.5 * (1 - torch.cos(math.pi * xx / e)), w)
        w = torch.where(xx > 1 - e, 0.5 * (1 - torch.cos(math.pi * (1 - xx) / e)), w)
        z = torch.fft.ifft(torch.fft.ifftshift(spec * w)) * no / math.sqrt(M * no)
        off = int(round(float(t[a]) / (t_len / n1)))
        out[off:off + no] = z * _cis(_f64(-(d.k_het / t_len) * float(t[a])))
        a = i
    return out


def _demod_exact(c, d, X, t, pd, tm):
    T = d.sft_len * d.dt_raw
    X = X.to(torch.complex128)
    n = pd.n_fft
    q = torch.arange(c["n_q"], dtype=torch.float64, device=DEV) + (n // 2 - c["n_q"] // 2)
    f = pd.f_het + (q - n // 2) / (n * pd.dt)
    mid = _f64(t) + T / 2
    out = []
    for rec in tm:
        al, de, fd = _f64(float(rec["alpha"])), _f64(float(rec["delta"])), float(rec["fdot"])
        tau = mid - pd.t_start + _delay(mid, al, de, pd)
        rate = _rate(mid, al, de, pd)
        a, b = _beams(mid, al, de, pd)
        Fa = torch.zeros(c["n_q"], dtype=torch.complex128, device=DEV)
        Fb = torch.zeros_like(Fa)
        for s in range(len(t)):
            kap = (f + fd * tau[s]) * (1 + rate[s]) * T
            ks = torch.floor(kap)
            S = torch.zeros_like(Fa)
            for j in range(-d.dirichlet_terms, d.dirichlet_terms + 1):
                y = TAU * (kap - ks - j)
                ys = torch.where(y == 0, 1.0, y)
                P = torch.complex(torch.where(y == 0, 1.0, torch.sin(y) / ys),
                                  torch.where(y == 0, 0.0, -(1 - torch.cos(y)) / ys))
                S += X[s, (ks.long() + j) - d.k_lo] * P
            ph = f * tau[s]
            w = S * _cis(-((ph - torch.round(ph)) + 0.5 * fd * tau[s] ** 2 - 0.5 * kap))
            Fa += a[s] * w
            Fb += b[s] * w
        out.append(_two_f(Fa, Fb, torch.ones_like(a), a, b, 1.0))
    return torch.stack(out)


def exact(case, seed):
    k = case["kind"]
    if k == "compute":
        d, x, t, gaps = _compute_inputs(case, seed)
        x = x.to(torch.complex128)
        band = (d.n_fft // 4, 3 * d.n_fft // 4) if case["half_band"] else None
        return torch.cat([_spectrum(x, i, gaps, d, d.n_fft, band) for i in t])
    if k == "ragged":
        d, x, t, gaps = _ragged_inputs(case, seed)
        x = x.to(torch.complex128)
        return torch.cat([_spectrum(x, i, gaps, d, int(i["n_fft"])) for i in t])
    if k == "montecarlo":
        d, x, inj, t = _mc_inputs(case, seed)
        x = x.to(torch.complex128)
        for i in inj:
            a = int(i["span_start"])
            x[a:a + int(i["span_len"])] += _signal(i, d)
        # 2F of the series that the search is given, in its own 32 bits
        xs = x.to(torch.complex64).to(torch.complex128)
        none = np.zeros((0, 2), np.int64)
        return {"x": x, "two_f": torch.cat([_spectrum(xs, i, none, d, d.n_fft) for i in t])}
    if k == "grad":
        d, x, t, gaps, theta = _grad_inputs(case, seed)
        x = x.to(torch.complex128)
        f, g = [], []
        for i in range(len(t)):
            th = theta[i].clone().requires_grad_()
            wa, wb, m, a, b, tau_b = _series(x, _valid(d, t[i], gaps), t[i], d, th)
            e = _cis(-th[2] * tau_b)
            v = _two_f((wa * e).sum(), (wb * e).sum(), m, a, b, d.sigma2)
            g.append(torch.autograd.grad(v, th)[0])
            f.append(v.detach())
        return {"two_f": torch.stack(f), "grad": torch.stack(g)}
    if k == "topk":
        f = _topk_input(case, seed).double().view(case["n_rows"], -1, case["band_len"])
        v, i = f.sort(dim=2, descending=True, stable=True)
        base = torch.arange(f.shape[1], device=DEV)[None, :, None] * case["band_len"]
        return [v[:, :, :case["k"]].contiguous(), (i[:, :, :case["k"]] + base).to(torch.int32)]
    if k == "sft":
        d, X, t = _sft_inputs(case, seed)
        return _sft_series_exact(d, X, t, case["slots"] * case["band_bins"])
    if k == "demod":
        return _demod_exact(case, *_demod_inputs(case, seed))
    d = Desc(n_data=case["n_inj"] * case["span"])
    inj = _injections(case["n_inj"], seed + 3, np.arange(case["n_inj"]) * case["span"], case["span"], 0.02)
    return torch.cat([_signal(i, d) for i in inj])
