"""The coefficient tables that the run kernels evaluate (sinc_run.cuh, demod.cu),
read from the sources and compared with the functions they stand for in 64
bits: the coefficients as written, that is rounded to single precision, and the
whole evaluation in single precision."""
import os
import re

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_0912_4255_gb300", "csrc")
G = np.linspace(-0.5, 0.5, 4001)


def _tables(name):
    src = open(os.path.join(CSRC, "sinc_run.cuh")).read()
    body = src[src.index(f"constexpr float {name}(int p, int k)"):]
    body = body[:body.index("return LANCZOS")]
    lz, rc = re.findall(r"constexpr float (?:lz|rc)\[4\]\[(?:\d+)\] = \{(.*?)\};", body, re.S)
    rows = [np.array([[float(v.rstrip("f")) for v in r.split(",")] for r in re.findall(r"\{([^{}]*)\}", t)])
            for t in (lz, rc)]
    return {"lanczos": rows[0], "rect": rows[1]}


def _sinc(x):
    """sin(pi x) / (pi x) and its first two derivatives."""
    x = np.where(np.abs(x) < 1e-2, np.nan, x)                 # removable singularity: not sampled
    s = np.sin(np.pi * x) / (np.pi * x)
    d = (np.cos(np.pi * x) - s) / x
    return s, d, (-np.pi * np.sin(np.pi * x) - 2 * d) / x


def _kernel(x, window):
    s, d, e = _sinc(x)
    if window == "rect":
        return s, d, e
    w, wd, we = _sinc(x / 4)
    wd, we = wd / 4, we / 16
    return s * w, d * w + s * wd, e * w + 2 * d * wd + s * we


# table, derivative, error of the fit as the source states it
@pytest.mark.parametrize("window", ["lanczos", "rect"])
@pytest.mark.parametrize("name,order,fit", [("sinc_c0", 0, 8e-10), ("sinc_c1", 1, 2e-5), ("sinc_c2", 2, 2e-2),
                                            ("sinc_d1", 1, 4e-8), ("sinc_d2", 2, 3e-4)])
def test_tap_weight_tables(window, name, order, fit):
    """Each coefficient as written is off by half a unit in its last place at most; the
    evaluation rounds each of its steps, whose terms stay below sum |c_k| / 2^k, once
    for the product and once for the sum."""
    tab = _tables(name)[window]
    assert tab.shape[0] == 4
    for p in range(4):
        # taps p and 7 - p from one polynomial: K(x_p) at g and K(x_{7-p}) = K_p(-g)
        for sign, x in ((1, G + 3.5 - p), (-1, G - 3.5 + p)):
            f = _kernel(x, window)[order] * (0.5 if order == 2 else 1.0) * (sign if order == 1 else 1)
            ok = np.isfinite(f)
            c = tab[p].astype(np.float32)
            half = 0.5 ** np.arange(len(c))
            bound = fit + np.sum(np.spacing(np.abs(c)) / 2 * half)
            got = np.polynomial.polynomial.polyval(sign * G, c.astype(np.float64))
            assert np.abs(got - f)[ok].max() < bound, (p, sign, np.abs(got - f)[ok].max())
            g = G.astype(np.float32)
            t = g * g
            even, odd = np.float32(0), np.float32(0)
            for k in range(len(c) - 1, -1, -1):
                if k % 2:
                    odd = odd * t + c[k]
                else:
                    even = even * t + c[k]
            got32 = even + np.float32(sign) * g * odd
            assert np.abs(got32 - f)[ok].max() < bound + 2 * 2.0 ** -24 * np.sum(np.abs(c) * half), (p, sign)


def test_demodulation_polynomials():
    """sin(pi x) / pi relative to the distance from 0 and 1, and sin, cos(pi v) on
    half a turn, with the coefficients as written."""
    src = open(os.path.join(CSRC, "demod.cu")).read()

    def horner(text, u):
        c = [float(v) for v in re.findall(r"(-?\d+\.\d+)f", text)]        # leading coefficient first
        r = np.zeros_like(u)
        for v in c:
            r = r * u + np.float64(np.float32(v))
        return r

    x = np.linspace(1e-6, 0.5, 20001)
    body = src[src.index("float sinpi_over_pi(float f)"):]
    poly = re.search(r"return x \* (fmaf.*);", body).group(1)
    assert np.abs(x * horner(poly, x * x) / (np.sin(np.pi * x) / np.pi) - 1).max() < 1.5e-8
    body = src[src.index("void sincospi_half("):]
    sn, cs = re.search(r"\*s = v \* (fmaf.*);", body).group(1), re.search(r"\*c = (fmaf.*);", body).group(1)
    assert np.abs(x * horner(sn, x * x) - np.sin(np.pi * x)).max() < 5e-8
    assert np.abs(horner(cs, x * x) - np.cos(np.pi * x)).max() < 3e-8


@pytest.mark.parametrize("window", ["lanczos", "rect"])
def test_interpolant_has_no_bias(window):
    """The mean error of the eight weights, evaluated in single precision, on a
    harmonic of any frequency of the band: what the coherent sum of 2F keeps of
    the weights' errors.  Below a quarter of the unit roundoff of single precision."""
    tab = _tables("sinc_c0")[window].astype(np.float32)
    g = np.random.default_rng(0).uniform(-0.5, 0.5, 200_001)
    g32 = g.astype(np.float32)
    t = g32 * g32

    def fma(a, b, c):
        return (a.astype(np.float64) * b + c).astype(np.float32)

    for om in (0.0, 0.1, 0.25):
        err, ideal = 0.0, 0.0
        for p in range(4):
            even, odd = np.full_like(t, tab[p][10]), np.full_like(t, tab[p][9])
            for k in (8, 6, 4, 2, 0):
                even = fma(even, t, tab[p][k])
            for k in (7, 5, 3, 1):
                odd = fma(odd, t, tab[p][k])
            for w, x in ((fma(g32, odd, even), g + 3.5 - p), (fma(-g32, odd, even), g - 3.5 + p)):
                k0 = np.sinc(x) * (np.sinc(x / 4) if window == "lanczos" else 1.0)
                e = np.exp(-2j * np.pi * om * x)
                err, ideal = err + (w - k0) * e, ideal + k0 * e
        assert abs(np.mean(err / ideal)) < 0.25 * 2.0 ** -24, om
