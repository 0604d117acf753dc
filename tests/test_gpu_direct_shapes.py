"""The direct pair sum's row kernel in every instance that its launch rule picks:
2 and 4 targets a thread (FP32), 2 (FP64), rows of one and of several target chunks, with
full and with partly filled last chunks.  Seeded cells and both ends of rows against the FP64
oracle's direct sum, at the tolerances of the parity tests.  (test_direct_tile.py holds the
sizes to the rule.)"""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu

TOL = {torch.float32: (1e-5, 1e-4), torch.float64: (1e-11, 1e-11)}
F32 = [(232, 97), (232, 128), (45, 521), (37, 768), (162, 326), (127, 768), (45, 1158), (85, 768)]
F64 = [(8, 8), (8, 326), (8, 768), (20, 256), (8, 225)]


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()
    oracle.build()


@pytest.mark.parametrize("nr,nphi,dtype", [(*s, torch.float32) for s in F32] + [(*s, torch.float64) for s in F64])
def test_every_instance(nr, nphi, dtype):
    from paper_2506_10812_gb300 import Plan
    rng = np.random.default_rng(17 * nr + nphi)
    npdt = np.float32 if dtype == torch.float32 else np.float64
    g = oracle.Grid(nr, nphi, 0.3, 3.0)
    R, P = g.mesh()
    sg, sd = rng.uniform(0.5, 1.5, R.shape).astype(npdt), rng.uniform(0.005, 0.015, R.shape).astype(npdt)
    Hg = (0.05 * R * (1 + 0.3 * np.cos(P))).astype(npdt)
    Hd = (0.01 * R * (1 + 0.3 * np.sin(3 * P))).astype(npdt)
    rows = np.array([0, nr // 2, nr - 1])
    ends = np.concatenate([rows * nphi, rows * nphi + nphi - 1, rows * nphi + nphi // 2])
    idx = np.unique(np.concatenate([ends, rng.choice(nr * nphi, min(60, nr * nphi), replace=False)])).astype(np.int64)
    ref = oracle.direct(g, sg.astype(float), sd.astype(float), H_g=Hg.astype(float), H_d=Hd.astype(float), G=1.0,
                        targets=idx)
    t = lambda a: torch.tensor(a, dtype=dtype, device="cuda:0")  # noqa: E731
    with Plan(nr, nphi, 0.3, 3.0, 0.05, 0.005, dtype=dtype, method="direct", H_g=t(Hg), H_d=t(Hd)) as pl:
        out = pl.solve(t(sg), t(sd))
        again = pl.solve(t(sg), t(sd))
        pl.sync()
    for k, v in out.items():
        assert torch.equal(v, again[k]), k
        d = v.double().cpu().numpy().ravel()[idx] - ref[k]
        scale = ref[k] if k.startswith("phi") else np.hypot(ref["gr" + k[-2:]], ref["gphi" + k[-2:]])
        assert np.linalg.norm(d) <= TOL[dtype][0] * np.linalg.norm(scale), k
        assert np.max(np.abs(d)) <= TOL[dtype][1] * np.max(np.abs(scale)), k
