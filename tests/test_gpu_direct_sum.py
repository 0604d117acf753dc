"""The direct sum's additions by themselves.  For scale heights far below the cells
both Bessel tails are 1 and a pair's potential is the product of two numbers that
are computed here exactly as the kernel computes them (a source's mass over
sqrt(r r') and a lag's 1 / sqrt(sigma)), so that what separates an output from the
exact sum of the exact products is the summation alone.

Bound: 0.36 units in the last place, root mean square.  Rounding a sum once is 0.29 (up to
0.33 by where in its binade the sum lies); rounding each product before it is added
leaves 0.29 / sqrt(n) units more; sums of 16 terms without compensation 0.5 and more."""
import math

import numpy as np
import pytest
import torch

from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu
R_IN, R_OUT = 0.5, 2.0


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()


def products(nr, nphi, sigma):
    """(masses, weights): factors of the pair's term for every row pair; arrays in sigma's type."""
    f = sigma.dtype.type
    du, dphi = math.log(R_OUT / R_IN) / nr, 2.0 * math.pi / nphi
    area = du * dphi
    c, c_lo = f(area), f(area - float(f(area)))
    r = np.array([R_IN * math.exp((i + 0.5) * du) for i in range(nr)], dtype=f)
    gi = {d: f(math.sinh(0.5 * (d * du)) ** 2) for d in range(-(nr - 1), nr)}
    sp = [math.sin(math.pi * min(d, nphi - d) / nphi) for d in range(nphi)]
    gj = np.array([s * s for s in sp], dtype=f)
    x = ((sigma * r[:, None]) * r[:, None]).astype(f)
    if f is np.float32:      # one rounding of the exact x c + round(x c_lo)
        mass = (x.astype(np.float64) * float(c) + (x * c_lo).astype(np.float64)).astype(f)
    else:
        mass = x * c
    out = []
    for i in range(nr):
        row = []
        for k in range(nr):
            q = f(1) / np.sqrt(r[i] * r[k])
            with np.errstate(divide="ignore"):
                w = f(1) / np.sqrt(f(4) * (gi[i - k] + gj))
            row.append((mass[k] * q, w))
        out.append(row)
    return out


def exact_sums(nr, nphi, sigma):
    from fractions import Fraction
    ref = np.empty((nr, nphi), dtype=object)
    for i, row in enumerate(products(nr, nphi, sigma)):
        pairs = [([Fraction(float(a)) for a in m], [Fraction(float(b)) if np.isfinite(b) else None for b in w])
                 for m, w in row]
        for j in range(nphi):
            ref[i, j] = sum(m[(j - d) % nphi] * w[d] for k, (m, w) in enumerate(pairs) for d in range(nphi)
                            if not (k == i and d == 0))
    return ref


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_terms_are_compensated(dtype):
    from paper_2506_10812_gb300 import Plan
    npdt = np.float32 if dtype == torch.float32 else np.float64
    err = []
    for nr, nphi in [(1, 24), (1, 40), (1, 63), (2, 33), (3, 20), (5, 17)]:
        sigma = np.random.default_rng(100 * nr + nphi).uniform(0.5, 1.5, (nr, nphi)).astype(npdt)
        H = torch.full((nr, nphi), 1e-7 if dtype == torch.float32 else 1e-12, dtype=dtype, device="cuda:0")
        with Plan(nr, nphi, R_IN, R_OUT, 0.05, dtype=dtype, method="direct", H_g=H) as pl:
            phi = pl.solve(torch.tensor(sigma, device="cuda:0"))["phi_g"].cpu().numpy()
        for v, e in zip(phi.ravel(), exact_sums(nr, nphi, sigma).ravel()):
            err.append(float(-e) and float((e + type(e)(float(v))) / type(e)(float(np.spacing(npdt(float(e)))))))
    err = np.array(err)
    assert np.abs(err).max() < 8, "the products are not the kernel's"
    assert np.sqrt(np.mean(err ** 2)) <= 0.36, np.sqrt(np.mean(err ** 2))
