"""FP32 rounding of the semi-spectral solve: noisy gas + dust discs on seven grids,
four flaring scale heights, against FP64 plans on the same FP32 inputs.  Mean relative
L2 errors.  Bounds: Phi and g_r as measured on these discs when a lane took two complex table
entries at a time (7.35e-8, 1.28e-7); g_phi, which was 1.795e-7 then and 1.827e-7 with
four entries in one chain of additions, 1.81e-7."""
import numpy as np
import pytest
import torch

from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu
BOUND = {"phi": 7.35e-8, "gr": 1.28e-7, "gphi": 1.81e-7}


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()


def test_errors():
    from paper_2506_10812_gb300 import Plan
    dev, means = torch.device("cuda:0"), {}
    for nr, nphi in [(16, 32), (32, 64), (64, 128), (64, 64), (128, 128), (128, 256), (256, 256)]:
        r = (0.1 * 50.0 ** ((np.arange(nr) + 0.5) / nr))[:, None]
        err = {}
        for h in (0.02, 0.04, 0.07, 0.12):
            Hg = torch.tensor(h * r ** 1.25 * np.ones((1, nphi)), dtype=torch.float32, device=dev)
            Hd = Hg * 0.1
            how = dict(method="semispectral")
            with Plan(nr, nphi, 0.1, 5.0, 0.05, 0.005, H_g=Hg, H_d=Hd, **how) as p32, \
                    Plan(nr, nphi, 0.1, 5.0, 0.05, 0.005, dtype=torch.float64, H_g=Hg.double(), H_d=Hd.double(), **how) as p64:
                for k in range(16):
                    s = np.random.default_rng(nr * 100 + k).uniform(0.5, 1.5, (nr, nphi)) / r
                    sg = torch.tensor(s, dtype=torch.float32, device=dev)
                    ref = p64.solve(sg.double(), (sg * 0.01).double())
                    for q, v in p32.solve(sg, sg * 0.01).items():
                        err.setdefault(q[:-2], []).append(float((v.double() - ref[q]).norm() / ref[q].norm()))
        for q, v in err.items():
            means.setdefault(q, []).append(np.mean(v))
    for q, v in means.items():
        assert np.mean(v) <= BOUND[q], (q, np.mean(v))
