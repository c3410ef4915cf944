"""The tiled kernels of the path at the sizes where they can go wrong: the
resampler in runs of eight points against the kernel that takes one point at a
time (persistent mode) and the oracle, the FFT passes at their extreme shapes,
the gradient in runs against the FP64 plan's point-by-point gradient, the
front end's running median and its transforms of every band length."""
import numpy as np
import pytest

import synth
from oracle import frontend as FE
from oracle import resample as R

from _gpu import MODES, injected_series, oracle_two_f, r15, run_compute, tie_margin

pytestmark = pytest.mark.gpu
TOL = 1e-4                       # R15 against the oracle, as everywhere


def _templates(desc, spans, n_gaps, seed, fdot=(-1e-9, 0.0), gap_free=True):
    """One template per (start, length); nearest neighbours no nearer to a tie
    than 1e-6 samples (positions are held to ~1e-8)."""
    g = synth.rng(seed)
    out = []
    for i, (s, n) in enumerate(spans):
        for _ in range(50):
            t = synth.make_templates(g.uniform(0, 2 * np.pi), np.arcsin(g.uniform(-1, 1)), g.uniform(*fdot), s, n, 0,
                                     0 if i == 0 and gap_free else n_gaps)
            if desc.interp != R.NEAREST or tie_margin(desc, t[0]) > 1e-6:
                break
        out.append(t)
    tm = np.concatenate(out)
    tm["out_off"] = np.arange(len(tm)) * desc.n_fft
    return tm


# n_data, n_fft, log2_n1 (N2 from 2^6 to 2^12), f_het, dt, knot_log2.  Every span
# covers six hours at least: over minutes a(t) and b(t) are nearly proportional,
# D = AB - C^2 nearly 0, and 2F magnifies the rounding of A, B, C by AB / D.  With
# long samples knots 32 apart keep a and b within 1e-6 between knots (the default
# spacing is for dt below a second or so).
SHAPES = [
    (3001, 1 << 12, 6, 20.0, 16.0, 5),
    (4001, 1 << 13, 7, 20.0, 16.0, 5),
    (8000, 1 << 13, 7, 100.0, 8.0, 5),
    (30011, 1 << 15, 6, 20.0, 2.0, 0),
    (30011, 1 << 15, 9, 1000.0, 2.0, 0),
    (65001, 1 << 17, 7, 1500.0, 1.0, 0),
    (65001, 1 << 17, 11, 100.0, 1.0, 6),
    (100_003, 1 << 17, 8, 100.0, 0.5, 4),
    (200_001, 1 << 18, 6, 300.0, 0.5, 0),
]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["nearest", "rect", "lanczos"])
def test_runs_of_eight_against_single_points_and_the_oracle(shape, kind):
    """Gaps of one sample, of odd lengths, next to each other but one and at
    the ends; spans that start and end at odd samples, one without gaps; the
    series at both 8-byte alignments, with NaN around it."""
    import torch
    import paper_0912_4255_gb300 as fs
    n_data, n_fft, l1, f_het, dt, knot = shape
    d = synth.PlanDesc(dt=dt, n_data=n_data, n_fft=n_fft, f_het=f_het, max_templates=4,
                       interp=R.NEAREST if kind == "nearest" else R.SINC,
                       window=R.WIN_RECT if kind == "rect" else R.WIN_LANCZOS)
    h = n_data // 2
    gaps = np.array([[0, 3], [101, 102], [103, 104], [111, 119], [h - 501, h + 4], [h + 7, h + 8], [h + 200, h + 777],
                     [n_data - 2, n_data]], np.int64)
    x, _ = injected_series(d, 31, [synth.random_injection(32, df=0.1 / dt)], gaps)
    tm = _templates(d, [(0, n_data), (0, n_data), (17, n_data - 40), (h // 2 - 3, h + 1)], len(gaps), 33)
    got, rc = run_compute(d, x, tm, gaps, mode=MODES["split"], tuning=dict(log2_n1=l1, knot_log2=knot))
    single, rc2 = run_compute(d, x, tm, gaps, mode=MODES["persistent"], tuning=dict(knot_log2=knot))
    assert rc == 0 and rc2 == 0
    for i in range(4):
        assert r15(got[i], single[i]) <= TOL, i
        assert r15(got[i], oracle_two_f(d, x, tm[i], gaps)) <= TOL, i
    # the same series eight bytes further
    dev = torch.device("cuda:0")
    plan = fs.Plan(d, device=dev)
    plan.set_tuning(mode=fs.MODE_SPLIT, log2_n1=l1, knot_log2=knot)
    both = []
    for off in (0, 1):
        buf = torch.full((n_data + 2,), float("nan"), dtype=torch.complex64, device=dev)
        buf[off:off + n_data] = torch.from_numpy(x).to(dev)
        both.append(fs.fstat_compute(plan, buf[off:off + n_data], fs.pack_templates(tm, device=dev),
                                     torch.from_numpy(gaps.reshape(-1).copy()).to(dev)))
    for a in both:
        assert r15(a.cpu().numpy().reshape(4, -1), got) <= TOL
    plan.close()


@pytest.mark.parametrize("l_fft,l1", [(12, 6), (14, 8), (16, 10), (18, 9), (18, 7), (19, 12), (20, 11), (20, 10), (21, 12),
                                      (21, 9), (22, 10), (24, 12)])
def test_fft_shapes(l_fft, l1):
    """First passes of 2^6 .. 2^12 with second passes of 2^6 .. 2^12, whole and
    half-empty series, two templates: every bin against the oracle."""
    n = 1 << l_fft
    d = synth.PlanDesc(dt=max(0.5, 65536 / n), n_data=n - n // 100 - 9, n_fft=n, f_het=40.0, max_templates=2,
                       interp=R.NEAREST)
    x = synth.complex_noise(d.n_data, 1.0, 40 + l_fft)
    tm = synth.make_templates([0.4, 2.2], [0.3, -0.8], [-1e-9, 0.0], [0, 777], [d.n_data, d.n_data // 2])
    got, rc = run_compute(d, x, tm, mode=MODES["split"], tuning=dict(log2_n1=l1, knot_log2=5 if d.dt > 2 else 0))
    assert rc == 0
    for i in range(2):
        # a nearest neighbour within the positions' error of a tie may go either
        # way: one sample of n changes 2F by at most a few |x| sqrt(2F / n)
        slack = 0.0 if tie_margin(d, tm[i]) > 1e-6 else 40.0 / np.sqrt(tm[i]["span_len"])
        assert r15(got[i], oracle_two_f(d, x, tm[i])) <= TOL + slack, i


@pytest.mark.parametrize("window", [R.WIN_LANCZOS, R.WIN_RECT])
@pytest.mark.parametrize("n_data,f_het,dt", [(3001, 20.0, 16.0), (90_001, 1000.0, 0.5)])
def test_fp64_weights(window, n_data, f_het, dt):
    """The FP64 8-tap weights, gaps and edges included (1e-6 as in the FP64
    test of the path)."""
    d = synth.PlanDesc(dt=dt, n_data=n_data, n_fft=1 << 17, interp=R.SINC, window=window, f_het=f_het,
                       precision=synth.PREC_FP64, max_templates=2)
    gaps = np.array([[0, 2], [500, 501], [503, 900], [n_data - 5, n_data]], np.int64)
    x, _ = injected_series(d, 51, [synth.random_injection(52, df=0.2 / dt)], gaps)
    tm = _templates(d, [(0, n_data), (9, n_data - 20)], len(gaps), 53, gap_free=False)
    for mode in ("split", "fused"):
        got, rc = run_compute(d, x, tm, gaps, mode=MODES[mode], tuning=dict(knot_log2=5 if dt > 2 else 0))
        assert rc == 0
        for i in range(2):
            assert r15(got[i], oracle_two_f(d, x, tm[i], gaps)) <= 1e-6


@pytest.mark.parametrize("window", [R.WIN_LANCZOS, R.WIN_RECT])
@pytest.mark.parametrize("n_data,dt,df,f_het", [(2050, 16.0, 0.04, 20.0),
                                                (5003, 8.0, -0.06, 100.0), (70_001, 1.0, 0.3, 1000.0)])
def test_gradient_runs_against_the_fp64_gradient(window, n_data, dt, df, f_het):
    """The FP32 gradient kernels (runs of eight) against the FP64 plan's, which
    takes one point at a time: 2F within 1e-4, the gradient within 1e-3 in
    the metric's scales (the tolerances of the adjoint's test)."""
    import torch
    import paper_0912_4255_gb300 as fs
    d = synth.PlanDesc(dt=dt, n_data=n_data, n_fft=synth.next_pow2(n_data + 64), interp=R.SINC, window=window,
                       f_het=f_het, max_templates=5)
    h = n_data // 2
    gaps = np.array([[0, 1], [9, 10], [12, 13], [h, h + n_data // 10], [n_data - 2, n_data]], np.int64)
    inj = synth.random_injection(61, df=df)
    x, _ = injected_series(d, 62, [inj], gaps)
    spans = [(0, n_data), (3, n_data - 7), (h // 2, h)]
    tm = np.concatenate([synth.make_templates(inj.alpha + 1e-3 * i, inj.delta, inj.fdot, s, n, 0, len(gaps))
                         for i, (s, n) in enumerate(spans)])
    dev = torch.device("cuda:0")
    out = []
    for prec in (synth.PREC_MIXED, synth.PREC_FP64):
        plan = fs.Plan(d.replace(precision=prec), device=dev)
        y, g = fs.fstat_grad(plan, torch.from_numpy(x).to(dev), fs.pack_templates(tm, device=dev),
                             torch.full((3,), df, dtype=torch.float64),
                             torch.from_numpy(gaps.reshape(-1).copy()).to(dev))
        assert fs.fstat_status(plan, raise_error=False) == 0
        out.append((y.cpu().numpy(), g.cpu().numpy()))
        plan.close()
    (y, g), (y64, g64) = out
    T = n_data * dt
    scale = np.array([1e-3, 1e-3, 1.0 / T, 1.0 / T ** 2])
    for i in range(3):
        assert abs(y[i] - y64[i]) / max(y64[i], 4.0) < 1e-4, i
        assert np.linalg.norm((g[i] - g64[i]) * scale) < 1e-3 * max(np.linalg.norm(g64[i] * scale),
                                                                    1e-3 * max(y64[i], 4.0)), i


@pytest.mark.parametrize("w", [1, 3, 63, 65, 127, 129, 255, 257, 1023])
def test_running_median(w):
    """Windows around the places per lane, bands shorter and longer than the
    window and than a warp's run, ties, zeros, in place."""
    import torch
    import paper_0912_4255_gb300 as fs
    for K in (1, 37, 64, 700, 1100):
        g = synth.rng(80 + w + K)
        X = (g.normal(size=(3, K)) + 1j * g.normal(size=(3, K))).astype(np.complex64)
        X[1] = np.round(X[1] * 2) / 2                # many equal powers, zeros among them
        sd = synth.SftDesc(sft_len=8192, dt_raw=1.0 / 32, k_lo=0, n_bins=K, k_het=K // 2, band_bins=2, dirichlet_terms=0,
                           median_window=w)
        t = torch.from_numpy(X).cuda()
        got = fs.fstat_sft_normalize(sd, t)
        want = FE.normalize(X.astype(np.complex128), w)
        ok = np.isfinite(want)                       # a window of zeros: zero here
        assert np.abs(got.cpu().numpy() - np.where(ok, want, 0))[ok].max() < 2e-5 * np.abs(want[ok]).max()
        assert torch.equal(fs.fstat_sft_normalize(sd, t, out=t), got)


@pytest.mark.parametrize("n1", [2, 6, 10, 26, 30, 32, 74, 90, 100, 162, 250, 256, 360, 900])
@pytest.mark.parametrize("n_slots", [1, 31, 33])
def test_band_lengths_and_chunk_lengths(n1, n_slots):
    """Band lengths with radices 4, 2, 3 and 5 and with other primes (26, 74),
    chunks around the tile of 32 SFTs: every sample against the oracle
    (tolerance as in the front end's test)."""
    import torch
    import paper_0912_4255_gb300 as fs
    N, dk = 4096, 4
    k_h = N // 4
    d = synth.SftDesc(sft_len=N, dt_raw=1.0 / 256.0, k_lo=k_h - n1 // 2 - dk - 2, n_bins=n1 + 2 * (dk + 2), k_het=k_h,
                      band_bins=n1, dirichlet_terms=dk)
    slots = np.arange(n_slots + 2)
    slots = np.delete(slots, n_slots)                # a chunk of n_slots and one of a single SFT
    g = synth.rng(90 + n1 + n_slots)
    X = (g.normal(size=(len(slots), d.n_bins)) + 1j * g.normal(size=(len(slots), d.n_bins))).astype(np.complex64)
    t = slots * d.t_sft
    n_out = (n_slots + 2) * n1
    want = FE.sft_to_series(X.astype(np.complex128), t, d, 0.0, n_out)
    got = fs.fstat_sft_series(d, torch.from_numpy(X).cuda(), t, 0.0, n_out).cpu().numpy()
    assert np.abs(got - want).max() < 3e-5 * np.abs(want).max()


@pytest.mark.parametrize("n_t,l_fft", [(1, 12), (1, 17), (64, 17), (65, 17), (2, 22)])
@pytest.mark.parametrize("mode", ["split", "fused", "plain"])
def test_calls_one_after_another(n_t, l_fft, mode):
    """Up to 2^23 points per launch the kernels of a call start while the one
    before still runs: calls on different series, eager and from a CUDA graph,
    without a pause between them give what each gives alone, bit for bit."""
    import torch
    import paper_0912_4255_gb300 as fs
    n = 1 << l_fft
    d = synth.PlanDesc(dt=max(0.5, 65536 / n), n_data=int(0.7 * n) | 1, n_fft=n, f_het=40.0, max_templates=n_t,
                       interp=R.SINC)
    dev = torch.device("cuda:0")
    plan = fs.Plan(d, device=dev)
    plan.set_tuning(mode=MODES[mode])
    g = synth.rng(95)
    tm = synth.make_templates(g.uniform(0, 6, n_t), g.uniform(-1, 1, n_t), g.uniform(-1e-9, 0, n_t), 0, d.n_data)
    tm = fs.pack_templates(tm, device=dev)
    xs = [torch.from_numpy(synth.complex_noise(d.n_data, 1.0, 96 + i)).to(dev) for i in range(3)]
    alone = []
    for x in xs:
        alone.append(fs.fstat_compute(plan, x, tm))
        torch.cuda.synchronize()
    outs = [torch.empty_like(a) for a in alone]

    def calls():
        for _ in range(2):
            for x, o in zip(xs, outs):
                fs.fstat_compute(plan, x, tm, twoF=o)

    calls()
    torch.cuda.synchronize()
    assert all(torch.equal(o, a) for o, a in zip(outs, alone))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for _ in range(2):
        for o in outs:
            o.zero_()
        graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(o, a) for o, a in zip(outs, alone))
    plan.close()


@pytest.mark.parametrize("n_sft,K", [(1, 200), (3, 932), (3, 3648), (320, 932), (3, 20000)])
def test_running_median_of_short_windows(n_sft, K):
    """Windows on both sides of the line between the two kernels, which moves
    with the number of SFTs and the band: against the oracle; with a NaN, an
    infinity and zeros in a row, every bin whose window has no NaN; a NaN counts
    above every number in both kernels; in place."""
    import torch
    import paper_0912_4255_gb300 as fs
    g = synth.rng(110 + K)
    X = (g.normal(size=(3, K)) + 1j * g.normal(size=(3, K))).astype(np.complex64)
    X[1] = np.round(X[1] * 2) / 2
    bad = K // 3
    X[2, bad] = np.nan
    X[2, bad + 70 if K > 400 else 0] = np.inf
    full = np.tile(X, ((n_sft + 2) // 3, 1))[:n_sft]
    for w in (1, 3, 7, 15, 21, 23, 31, 35, 45, 51, 61, 63):
        sd = synth.SftDesc(sft_len=8192, dt_raw=1.0 / 32, k_lo=0, n_bins=K, k_het=K // 2, band_bins=2, dirichlet_terms=0,
                           median_window=w)
        t = torch.from_numpy(full).cuda()
        got = fs.fstat_sft_normalize(sd, t)
        assert torch.equal(torch.nan_to_num(fs.fstat_sft_normalize(sd, t, out=t), 7.0), torch.nan_to_num(got, 7.0))
        got = got.cpu().numpy()
        for i in range(min(3, n_sft)):
            with np.errstate(invalid="ignore", over="ignore", divide="ignore"):
                p = np.abs(X[i].astype(np.complex128)) ** 2
                med = np.array([np.sort(p[max(0, k - w // 2):k + w // 2 + 1])[(len(p[max(0, k - w // 2):k + w // 2 + 1]) - 1) // 2]
                                for k in range(K)])                                # (NaN sorts last)
                want = X[i] * np.where(med > 0, 1 / np.sqrt(med / np.log(2.0)), 0)
            ok = np.isfinite(want)
            assert ok.sum() >= K - 2 * w - 2 and np.abs(got[i] - want)[ok].max() < 2e-5 * np.abs(want[ok]).max(), (w, i)
            assert np.array_equal(got[i::3], np.broadcast_to(got[i], got[i::3].shape), equal_nan=True)


def _orbit(speed):
    return synth.Ephem(au_m=synth.Ephem.au_m * speed)


@pytest.mark.parametrize("speed", [2.0, 4.2, 8.0])
@pytest.mark.parametrize("kind", ["nearest", "rect", "lanczos"])
def test_runs_on_a_faster_orbit(speed, kind):
    """Beyond 1.25 times the Earth's speed the runs' weights keep their square in
    the offset, beyond about 4.3 a run's offset leaves the expansion and its points
    are taken one by one, at 4.2 both happen in one call: every bin against the
    oracle, gaps included."""
    d = synth.PlanDesc(dt=1.0, n_data=120_001, n_fft=1 << 17, f_het=50.0, eph=_orbit(speed), max_templates=2,
                       interp=R.NEAREST if kind == "nearest" else R.SINC,
                       window=R.WIN_RECT if kind == "rect" else R.WIN_LANCZOS)
    gaps = np.array([[5000, 5003], [5010, 9000], [70_000, 70_001]], np.int64)
    x, _ = injected_series(d, 121, [synth.random_injection(122, df=0.1)], gaps)
    tm = _templates(d, [(0, d.n_data), (1001, 100_000)], len(gaps), 123, gap_free=False)
    got, rc = run_compute(d, x, tm, gaps, mode=MODES["split"], tuning=dict(knot_log2=6))
    assert rc == 0
    for i in range(2):
        assert r15(got[i], oracle_two_f(d, x, tm[i], gaps)) <= TOL, i


@pytest.mark.parametrize("speed", [2.0, 4.2, 8.0])
@pytest.mark.parametrize("window", [R.WIN_LANCZOS, R.WIN_RECT])
def test_gradient_runs_on_a_faster_orbit(window, speed):
    """The same for the gradient's runs, against the FP64 plan's gradient; the
    tolerances of the test on the Earth's orbit."""
    import torch
    import paper_0912_4255_gb300 as fs
    n, df = 90_001, 0.2
    d = synth.PlanDesc(dt=1.0, n_data=n, n_fft=1 << 17, interp=R.SINC, window=window, f_het=50.0, eph=_orbit(speed),
                       max_templates=2)
    gaps = np.array([[9, 10], [40_000, 44_001]], np.int64)
    inj = synth.random_injection(124, df=df)
    x, _ = injected_series(d, 125, [inj], gaps)
    tm = synth.make_templates([inj.alpha, inj.alpha + 1e-4], [inj.delta] * 2, [inj.fdot] * 2, [0, 77], [n, n - 1000], 0,
                              len(gaps))
    dev = torch.device("cuda:0")
    out = []
    for prec in (synth.PREC_MIXED, synth.PREC_FP64):
        plan = fs.Plan(d.replace(precision=prec), device=dev)
        plan.set_tuning(knot_log2=6)
        y, g = fs.fstat_grad(plan, torch.from_numpy(x).to(dev), fs.pack_templates(tm, device=dev),
                             torch.full((2,), df, dtype=torch.float64), torch.from_numpy(gaps.reshape(-1).copy()).to(dev))
        assert fs.fstat_status(plan, raise_error=False) == 0
        out.append((y.cpu().numpy(), g.cpu().numpy()))
        plan.close()
    (y, g), (y64, g64) = out
    T = n * d.dt
    scale = np.array([1e-3, 1e-3, 1.0 / T, 1.0 / T ** 2])
    for i in range(2):
        assert abs(y[i] - y64[i]) / max(y64[i], 4.0) < 1e-4, i
        assert np.linalg.norm((g[i] - g64[i]) * scale) < 1e-3 * max(np.linalg.norm(g64[i] * scale),
                                                                    1e-3 * max(y64[i], 4.0)), i


@pytest.mark.parametrize("l_fft,l1,prec", [(12, 6, 0), (14, 8, 0), (18, 12, 0), (18, 6, 0), (20, 8, 0), (21, 9, 0), (21, 12, 0),
                                           (22, 10, 0), (24, 12, 0), (12, 6, 1), (18, 12, 1), (18, 6, 1), (20, 10, 1)])
def test_fft_shapes_without_ties(l_fft, l1, prec):
    """The passes at their extreme shapes with the 8-tap sinc, which has no ties,
    so that every bin is held to the path's tolerance; the intermediate by row
    groups (split) and in place (fused)."""
    n = 1 << l_fft
    dt = max(0.5, 65536 / n)
    d = synth.PlanDesc(dt=dt, n_data=n - n // 50 - 9, n_fft=n, f_het=20.0, max_templates=1, interp=R.SINC,
                       precision=synth.PREC_FP64 if prec else synth.PREC_MIXED)
    x = synth.complex_noise(d.n_data, 1.0, 130 + l_fft)
    tm = synth.make_templates(0.4, 0.3, -1e-10, 0, d.n_data)
    want = oracle_two_f(d, x, tm[0])
    knot = 5 if dt > 2 else 7 if prec else 0
    for mode in ("split", "fused"):
        got, rc = run_compute(d, x, tm, mode=MODES[mode], tuning=dict(log2_n1=l1, knot_log2=knot))
        assert rc == 0
        assert r15(got[0], want) <= (1e-6 if prec else TOL), mode
