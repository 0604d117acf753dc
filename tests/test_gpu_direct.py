"""The direct pair sum's row decomposition at the sizes where it changes: short
rows, lag tiles (128 lags) that are exact, one over and one short, rows of
several target chunks, odd sizes, row counts below and above a cluster's
split; and scale heights from a thousandth of to ten times the radius, so that
every Bessel branch (series, tables, tails) is met.  Against the FP64 oracle's
direct sum, at the tolerances of the parity tests."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu

TOL = {torch.float32: (1e-5, 1e-4), torch.float64: (1e-11, 1e-11)}
SIZES = [(1, 9), (2, 8), (9, 7), (40, 3), (3, 127), (4, 128), (5, 129), (3, 257), (2, 1025), (17, 33), (23, 61)]


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()
    oracle.build()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nr,nphi", SIZES)
def test_row_decomposition(nr, nphi, dtype):
    from paper_2506_10812_gb300 import Plan
    rng = np.random.default_rng(1000 * nr + nphi)
    npdt = np.float32 if dtype == torch.float32 else np.float64
    g = oracle.Grid(nr, nphi, 0.3, 3.0)
    R, _ = g.mesh()
    sg, sd = rng.uniform(0.5, 1.5, R.shape).astype(npdt), rng.uniform(0.005, 0.015, R.shape).astype(npdt)
    # log-uniform per cell; a row of the gas is uniformly thin, so that whole rows take the tail
    Hg = R * 10.0 ** rng.uniform(-2.0, 1.0, R.shape)
    Hg[nr // 2] = R[nr // 2] * 1e-3
    Hd = R * 10.0 ** rng.uniform(-3.0, -1.0, R.shape)
    Hg, Hd = Hg.astype(npdt), Hd.astype(npdt)
    ref = oracle.direct(g, sg.astype(float), sd.astype(float), H_g=Hg.astype(float), H_d=Hd.astype(float), G=1.0)
    dev = torch.device("cuda:0")
    t = lambda a: torch.tensor(a, dtype=dtype, device=dev)  # noqa: E731
    with Plan(nr, nphi, 0.3, 3.0, 0.05, 0.005, dtype=dtype, method="direct", H_g=t(Hg), H_d=t(Hd)) as pl:
        out = pl.solve(t(sg), t(sd))
        again = pl.solve(t(sg), t(sd))
        pl.sync()
        for k, v in out.items():
            assert torch.equal(v, again[k]), k                  # ranks are added in a fixed order
            x = v.double().cpu().numpy()
            # fields are compared on the scale of their fluid's acceleration: g_phi of a few cells can cancel to nothing
            scale = ref[k] if k.startswith("phi") else np.hypot(ref["gr" + k[-2:]], ref["gphi" + k[-2:]])
            d = x - ref[k]
            assert np.linalg.norm(d) <= TOL[dtype][0] * np.linalg.norm(scale), k
            assert np.max(np.abs(d)) <= TOL[dtype][1] * np.max(np.abs(scale)), k
