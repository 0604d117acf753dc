"""FP64 transforms of every length (each final radix, one to four passes, rows
and columns) through the FFT solve, gas + dust, against the oracle's FP64
convolution at the FP64 tolerance of the parity tests."""
import pytest
import torch

import oracle
from paper_2506_10812_gb300 import build as B
from paper_2506_10812_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()
    oracle.build()


@pytest.mark.parametrize("nr,nphi", [(8, 32), (16, 64), (32, 8192), (64, 256), (128, 512), (256, 128), (512, 1024), (1024, 2048),
                                     (16, 4096)])
def test_every_length(nr, nphi):
    from paper_2506_10812_gb300 import Plan
    d = inputs.ragged_noise(nr, nphi, bifluid=True, offset=5 + nr)
    ref = oracle.fft64(oracle.Grid(nr, nphi, d.r_in, d.r_out), d.sigma_g, d.sigma_d, h_g=d.h_g, h_d=d.h_d, G=d.G)
    dev = torch.device("cuda:0")
    with Plan(nr, nphi, d.r_in, d.r_out, d.h_g, d.h_d, G=d.G, dtype=torch.float64) as pl:
        out = pl.solve(torch.tensor(d.sigma_g, device=dev), torch.tensor(d.sigma_d, device=dev))
        pl.sync()
        for k, v in out.items():
            x = v.cpu().numpy()
            assert oracle.rel_l2(x, ref[k]) <= 1e-11 and oracle.rel_max(x, ref[k]) <= 1e-11, k
