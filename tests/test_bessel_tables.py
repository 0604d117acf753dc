"""The committed Bessel coefficients (csrc/sg_bessel_tab.cuh) against the
oracle's functions, evaluated as the kernels do: entry and argument from the
bits of x, Horner's rule in the table's type.

Bounds: FP64, the fit (1.4e-17) plus Horner's few roundings, within the 2e-14
to which the oracle itself is pinned; FP32, the fit (1.3e-8) plus about three
roundings of 6e-8."""
import os
import re

import numpy as np

import oracle

PATH = os.path.join(os.path.dirname(__file__), "..", "paper_2506_10812_gb300", "csrc", "sg_bessel_tab.cuh")


def arrays():
    text = open(PATH).read()
    out = {}
    for name, body in re.findall(r"(BT_\w+)\[[^=]*= \{(.*?)\};", text, re.S):
        toks = re.findall(r"[-+]?0x[0-9a-fp.+-]+|[-+]?\d[\d.e+-]*", body)
        out[name] = np.array([float.fromhex(t) if "0x" in t else float(t) for t in toks])
    return out


def horner(c, t):
    acc = c[..., -1]
    for k in range(c.shape[-1] - 2, -1, -1):
        acc = (acc * t + c[..., k]).astype(t.dtype)
    return acc


def test_tables_and_tails():
    oracle.build()
    T = arrays()
    rng = np.random.default_rng(7)
    for dt, tab, n, tol in ((np.float64, "BT_64", 13, 3e-14), (np.float32, "BT_32", 6, 3e-7)):
        c = T[tab].astype(dt).reshape(96, 2, n)
        x = np.concatenate([2.0 ** rng.uniform(-20, 4, 20000), 2.0 ** np.arange(-20, 4)]).astype(dt)
        x = x[(x >= 2.0 ** -20) & (x < 16)]
        m, e = np.frexp(x)
        m, e = (2 * m).astype(dt), e - 1
        s = np.floor((m - 1) * 4).astype(int)
        t = (m - (1 + (2 * s + 1) / 8)).astype(dt)
        ent = c[4 * (e + 20) + s]
        k0, D = oracle.k0e_D(x.astype(np.float64))
        assert np.max(np.abs(horner(ent[:, 0], t) / k0 - 1)) < tol
        assert np.max(np.abs(horner(ent[:, 1], t) / (D * x.astype(np.float64)) - 1)) < tol
    z = rng.uniform(1e-9, 0.0625, 20000)
    for dt, sfx, tol in ((np.float64, "64", 3e-14), (np.float32, "32", 3e-7)):
        zz = z.astype(dt)
        x = 1.0 / zz.astype(np.float64)
        k0, D = oracle.k0e_D(x)
        w = np.sqrt(2 * x / np.pi)
        one = np.ones((zz.size, 1), dt)
        assert np.max(np.abs(horner(one * T["BT_S0_" + sfx].astype(dt), zz) / (k0 * w) - 1)) < tol
        assert np.max(np.abs(horner(one * T["BT_Q_" + sfx].astype(dt), zz) / (2 * D * x * w) - 1)) < tol
