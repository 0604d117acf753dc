"""FP32 rounding of the direct sum, against FP64 plans on the same FP32 inputs."""
import math

import numpy as np
import pytest
import torch

from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()


def solve_both(nr, nphi, sigma, H):
    from paper_2506_10812_gb300 import Plan
    s, h = (torch.tensor(a * np.ones((nr, nphi)), dtype=torch.float32, device="cuda:0") for a in (sigma, H))
    out = []
    for x, y in ((s, h), (s.double(), h.double())):
        with Plan(nr, nphi, 0.1, 5.0, 0.05, dtype=x.dtype, method="direct", H_g=y) as pl:
            out.append({k: v.double() for k, v in pl.solve(x).items()})
    return out


def disc(nr, nphi, h):
    """Surface density (20 % noise) and an azimuthally modulated scale height."""
    r = (0.1 * 50.0 ** ((np.arange(nr) + 0.5) / nr))[:, None]
    phi = (np.arange(nphi) + 0.5) * (2 * math.pi / nphi)
    noise = np.random.default_rng(nr * nphi).uniform(0.8, 1.2, (nr, nphi))
    return noise / r, h * r ** 1.25 * (1 + 0.15 * np.cos(phi + 1) + 0.05 * np.cos(3 * phi + 2))


def test_thick_discs():
    """Mean relative L2 error of the potential of discs half as thick as their radius,
    where two thirds of the pairs have X < 1.  Bound: 3.93e-8, measured on these discs
    with the Bessel functions of X < 1 evaluated in FP64 (FP32 tables: 5.81e-8)."""
    err = []
    for nr, nphi in [(24, 48), (61, 150), (45, 333), (97, 320), (200, 60)]:
        a, b = solve_both(nr, nphi, *disc(nr, nphi, 0.5))
        err.append(float((a["phi_g"] - b["phi_g"]).norm() / b["phi_g"].norm()))
    assert np.mean(err) <= 3.93e-8, err


def test_no_common_factor():
    """Relative offset of the potential as a whole, on grids whose cell area du dphi
    rounds to FP32 with an error of 5e-8 or more, thin and thick discs.  What all pairs
    share would show in full; independent roundings of 6e-8 average out to less than
    1.5e-8 over 28 rows and more."""
    worst = 0.0
    for nr, nphi in [(39, 80), (49, 64), (55, 112), (28, 112), (65, 96)]:
        area = math.log(50.0) / nr * 2 * math.pi / nphi
        assert abs(float(np.float32(area)) / area - 1) >= 5e-8, (nr, nphi)
        for h in (0.03, 0.5):
            a, b = solve_both(nr, nphi, *disc(nr, nphi, h))
            a, b = a["phi_g"], b["phi_g"]
            worst = max(worst, abs(float((a * b).sum() / (b * b).sum()) - 1))
    assert worst <= 1.5e-8
