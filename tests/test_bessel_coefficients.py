"""The committed Bessel coefficients (csrc/sg_bessel_tab.cuh) against K0 and K1 to
40 digits, at the accuracy that the file states: the polynomials that the
coefficients are, evaluated exactly, and the FP32 evaluation of the kernels (which adds the
rest of each polynomial to its rounded first coefficient) operation by operation.

Bounds.  FP64: the fits (1.4e-17) plus the coefficients' own rounding (2^-53 of the
first, an eighth of that of the second, and so on); tails 1.0e-16 and 1.3e-16.
FP32 tables with their remainders: 3e-9; their evaluation: the last addition's half
unit (2^-24) and the rest's three roundings, each of at most 0.15 of that.
FP32 tails: 6.4e-10 and 6.0e-9."""
import os
import re

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

PATH = os.path.join(os.path.dirname(__file__), "..", "paper_2506_10812_gb300", "csrc", "sg_bessel_tab.cuh")


def arrays():
    out = {}
    for name, body in re.findall(r"(BT_\w+)\[[^=]*= \{(.*?)\};", open(PATH).read(), re.S):
        toks = re.findall(r"[-+]?0x[0-9a-fp.+-]+|[-+]?\d[\d.e+-]*", body)
        out[name] = np.array([float.fromhex(t) if "0x" in t else float(t) for t in toks])
    return out


def k0e(x):
    return mp.exp(x) * mp.besselk(0, x)


def E(x):
    return x * mp.exp(x) * (mp.besselk(1, x) - mp.besselk(0, x))


def poly(c, t):
    return mp.polyval([mp.mpf(float(v)) for v in c[::-1]], t)


@pytest.fixture(autouse=True)
def digits():
    with mp.workdps(40):
        yield


def test_tables():
    T = arrays()
    t64, t32 = T["BT_64"].reshape(96, 2, 13), T["BT_32"].reshape(96, 2, 6)
    l32 = T["BT_32L"].reshape(96, 2, 2)
    for entry in range(96):
        e, s = entry // 4 - 20, entry % 4
        mid = mp.mpf(1) + mp.mpf(2 * s + 1) / 8
        for t in (mp.mpf(-1) / 8, mp.mpf(-1) / 11, mp.mpf(-1) / 70, mp.mpf(1) / 23, mp.mpf(1) / 9):
            x = (mid + t) * mp.mpf(2) ** e
            u2 = 64 * t * t
            T6 = ((32 * u2 - 48) * u2 + 18) * u2 - 1
            for q, f in enumerate((k0e, E)):
                ref = f(x)
                assert abs(poly(t64[entry, q], t) / ref - 1) < 1.4e-17 + 1.2 * 2.0 ** -53, (entry, q)
                got = poly(t32[entry, q], t) + mp.mpf(float(l32[entry, q, 0])) + mp.mpf(float(l32[entry, q, 1])) * T6
                assert abs(got / ref - 1) < 4e-9, (entry, q)


def test_tails():
    T = arrays()
    for i in range(1, 33):
        z = mp.mpf(i) / 512
        w = mp.sqrt(2 / (mp.pi * z))
        for name, ref, t64, t32 in (("S0", k0e(1 / z) * w, 1.05e-16, 6.5e-10), ("Q", 2 * E(1 / z) * w, 1.35e-16, 6.1e-9)):
            assert abs(poly(T[f"BT_{name}_64"], z) / ref - 1) < t64
            assert abs(poly(T[f"BT_{name}_32"], z) / ref - 1) < t32


def test_fp32_evaluation():
    f, d = np.float32, np.float64
    fma = lambda a, b, c: f(d(a) * d(b) + d(c))  # noqa: E731  (the FP64 sum's own rounding is 2^-29 of FP32's)
    T = arrays()
    t32, l32 = T["BT_32"].astype(f).reshape(96, 2, 6), T["BT_32L"].astype(f).reshape(96, 2, 2)
    rng = np.random.default_rng(3)
    worst = 0.0
    for _ in range(1500):
        x = f(2.0 ** rng.uniform(-20, 4))
        m, e = np.frexp(x)
        m, e = f(2 * m), e - 1
        s = int((m - 1) * 4)
        t = f(m - f(1 + (2 * s + 1) / 8))
        entry = 4 * (e + 20) + s
        v = f(f(64) * t) * t
        T6 = fma(fma(fma(f(32), v, f(-48)), v, f(18)), v, f(-1))
        for q, fn in enumerate((k0e, E)):
            c = t32[entry, q]
            r = c[5]
            for k in (4, 3, 2, 1):
                r = fma(r, t, c[k])
            got = f(c[0] + fma(r, t, fma(l32[entry, q, 1], T6, l32[entry, q, 0])))
            worst = max(worst, float(abs(mp.mpf(float(got)) / fn(mp.mpf(float(x))) - 1)))
    assert worst < 2.0 ** -24 * (1 + 3 * 0.15) + 4e-9
