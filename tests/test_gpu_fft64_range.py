"""FP64 solves near the top of the number range.  Scaling the surface density by a
power of two scales every rounding with it, so the outputs are those of the
unscaled disc times the same power, bit for bit, as long as nothing
overflows: 2^975 (3e293) times densities of order one leaves the sums of the
longest rows and columns here (2^25 terms) below 2^1024, and the transforms'
factors have to as well.  Every final radix and one to four passes."""
import pytest
import torch

from paper_2506_10812_gb300 import build as B
from paper_2506_10812_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()


@pytest.mark.parametrize("nr,nphi", [(8, 32), (16, 64), (64, 128), (128, 256), (256, 512), (1024, 1024), (32, 8192)])
def test_scaling_by_a_power_of_two_is_exact(nr, nphi):
    from paper_2506_10812_gb300 import Plan
    d = inputs.ragged_noise(nr, nphi, bifluid=True, offset=40 + nr)
    dev = torch.device("cuda:0")
    sg, sd = (torch.tensor(a, dtype=torch.float64, device=dev) for a in (d.sigma_g, d.sigma_d))
    with Plan(nr, nphi, d.r_in, d.r_out, d.h_g, d.h_d, G=d.G, dtype=torch.float64) as pl:
        out = pl.solve(sg, sd)
        big = pl.solve(sg * 2.0 ** 975, sd * 2.0 ** 975)
        for k, v in out.items():
            assert torch.equal(big[k], v * 2.0 ** 975), k
