"""The rounding of column 0, which carries the axisymmetric part of a disc and
dominates g_r: axisymmetric discs (every other column is zero) of 128 to 2048
rows, random from row to row, gas and gas + dust, FP32 against FP64 plans.

Bound: 1.88e-7 in the mean over these discs, on which column transforms that load
every root measured 1.868e-7 and ones that form nine of 15 as products 1.93e-7."""
import numpy as np
import pytest
import torch

from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()


def test_axisymmetric_discs():
    from paper_2506_10812_gb300 import Plan
    dev, nphi, means = torch.device("cuda:0"), 64, []
    for nr, h_d in [(n, h) for n in (128, 256, 512, 1024) for h in (None, 0.005)] + [(2048, None)]:
        r = 0.1 * 50.0 ** ((np.arange(nr) + 0.5) / nr)
        err = []
        with Plan(nr, nphi, 0.1, 5.0, 0.05, h_d) as p32, Plan(nr, nphi, 0.1, 5.0, 0.05, h_d, dtype=torch.float64) as p64:
            for k in range(32):
                s = np.random.default_rng(1000 * nr + k).uniform(0.5, 1.5, nr) / r
                sg = torch.tensor(s[:, None] * np.ones((1, nphi)), dtype=torch.float32, device=dev)
                sd = 0.01 * sg if h_d else None
                ref = p64.solve(sg.double(), None if sd is None else sd.double())
                for q, v in p32.solve(sg, sd).items():
                    if q.startswith("gr"):
                        err.append(float((v.double() - ref[q]).norm() / ref[q].norm()))
        means.append(np.mean(err))
    assert np.mean(means) <= 1.88e-7, means
