"""The column pass on both sides of its launch rules: grids whose (column,
output) CTAs fit the chip at once (split launches) and grids whose do not, short
rows and columns with compiled lengths, column 0 by output, row launches with
fewer CTAs than SMs.  Every output of a full solve equals the solve that asks
for it alone bit for bit, twice in a row, and the full solve meets the oracle at
the parity tests' tolerances."""
import pytest
import torch

import oracle
from paper_2506_10812_gb300 import build as B
from paper_2506_10812_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL = {torch.float32: (1e-5, 1e-4), torch.float64: (1e-11, 1e-11)}
COMPS = ("phi", "gr", "gphi")


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()
    oracle.build()


@pytest.mark.parametrize("bifluid", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nr,nphi", [(8, 32), (32, 64), (64, 128), (64, 512), (128, 256), (256, 512), (512, 512), (512, 1024)])
def test_outputs_do_not_depend_on_the_launch(nr, nphi, dtype, bifluid):
    from paper_2506_10812_gb300 import Plan
    d = inputs.ragged_noise(nr, nphi, bifluid=bifluid, offset=900 + nr)
    dev = torch.device("cuda:0")
    t = lambda a: None if a is None else torch.tensor(a, dtype=dtype, device=dev)  # noqa: E731
    sg, sd = t(d.sigma_g), t(d.sigma_d)
    h = lambda a: None if a is None else a.double().cpu().numpy()  # noqa: E731
    ref = oracle.fft64(oracle.Grid(nr, nphi, d.r_in, d.r_out), h(sg), h(sd), h_g=d.h_g, h_d=d.h_d, G=d.G)
    with Plan(nr, nphi, d.r_in, d.r_out, d.h_g, d.h_d, G=d.G, dtype=dtype) as pl:
        full = pl.solve(sg, sd)
        again = pl.solve(sg, sd)
        for c in COMPS:
            for k, v in pl.solve(sg, sd, outputs=(c,)).items():
                assert torch.equal(v, full[k]) and torch.equal(again[k], full[k]), k
        pl.sync()
        for k, v in full.items():
            x = v.double().cpu().numpy()
            assert oracle.rel_l2(x, ref[k]) <= TOL[dtype][0] and oracle.rel_max(x, ref[k]) <= TOL[dtype][1], k
