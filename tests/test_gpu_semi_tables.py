"""The semi-spectral tables at the edges of their decomposition: the shortest and
the longest rows (one row per CTA, and as many as there are radial cells), the
fewest radial cells (a part of a mode product's rows), in both types; scale heights
from a thousandth of to ten times the radius (every Bessel branch).  Against
the oracle's direct sum with the same heights, whole grids or seeded cells, at
the method's tolerances."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu

TOL = {torch.float32: (1e-5, 1e-4), torch.float64: (1e-11, 1e-11)}


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()
    oracle.build()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nr,nphi", [(8, 32), (8, 64), (32, 32), (64, 256), (16, 512), (8, 8192)])
def test_edges(nr, nphi, dtype):
    from paper_2506_10812_gb300 import Plan
    rng = np.random.default_rng(100 * nr + nphi)
    npdt = np.float32 if dtype == torch.float32 else np.float64
    g = oracle.Grid(nr, nphi, 0.3, 3.0)
    R, _ = g.mesh()
    sg, sd = rng.uniform(0.5, 1.5, R.shape).astype(npdt), rng.uniform(0.005, 0.015, R.shape).astype(npdt)
    Hg = (R * np.logspace(-2, 1, nr)[:, None]).astype(npdt)      # constant along phi
    Hd = (R * np.logspace(-1, -3, nr)[:, None]).astype(npdt)
    idx = np.arange(nr * nphi) if nr * nphi <= 2048 else np.sort(rng.choice(nr * nphi, 64, replace=False))
    ref = oracle.direct(g, sg.astype(float), sd.astype(float), H_g=Hg.astype(float), H_d=Hd.astype(float), G=1.0,
                        targets=None if idx.size == nr * nphi else idx.astype(np.int64))
    dev = torch.device("cuda:0")
    t = lambda a: torch.tensor(a, dtype=dtype, device=dev)  # noqa: E731
    with Plan(nr, nphi, 0.3, 3.0, 0.05, 0.005, dtype=dtype, method="semispectral", H_g=t(Hg), H_d=t(Hd)) as pl:
        out = pl.solve(t(sg), t(sd))
        pl.sync()
        for k, v in out.items():
            x, y = v.double().cpu().numpy().ravel()[idx], np.asarray(ref[k]).ravel()
            # on the scale of the fluid's acceleration, as g_phi of noise is small beside g_r
            a = y if k.startswith("phi") else np.hypot(*(np.asarray(ref[c + k[-2:]]).ravel() for c in ("gr", "gphi")))
            assert np.linalg.norm(x - y) <= TOL[dtype][0] * np.linalg.norm(a), k
            assert np.max(np.abs(x - y)) <= TOL[dtype][1] * np.max(np.abs(a)), k
