"""Direct plans whose scale-height field holds zeros.  A pair of two cells of
zero height has no kernel: every target of zero height that meets another such
cell is NaN in all outputs, and the finite check reports it; all other targets
are ordinary numbers, equal to the oracle's at the tolerances of the parity
tests.  Short rows (one thread per target) and long ones (row pairs) alike."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_10812_gb300 import _native as N
from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu

TOL = {torch.float32: 1e-5, torch.float64: 1e-11}


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()
    oracle.build()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("pattern", ["everywhere", "a row", "two cells", "one cell"])
@pytest.mark.parametrize("nphi", [5, 16, 300])
def test_zero_heights(nphi, pattern, dtype):
    from paper_2506_10812_gb300 import Plan
    nr = 6
    npdt = np.float32 if dtype == torch.float32 else np.float64
    g = oracle.Grid(nr, nphi, 0.3, 3.0)
    R, _ = g.mesh()
    H = (0.05 * R).astype(npdt)
    if pattern == "everywhere":
        H[:] = 0
    elif pattern == "a row":
        H[1] = 0
    elif pattern == "two cells":
        H[2, 3] = H[4, 1] = 0
    else:
        H[2, 3] = 0
    flat = H == 0
    none = flat & (flat.sum() > 1)               # the self cell is no pair
    sig = np.random.default_rng(nphi).uniform(0.5, 1.5, R.shape).astype(npdt)
    t = lambda a: torch.tensor(a, dtype=dtype, device="cuda:0")  # noqa: E731
    with Plan(nr, nphi, 0.3, 3.0, 0.05, dtype=dtype, method="direct", H_g=t(H), check_finite=True) as pl:
        out = {k: v.double().cpu().numpy() for k, v in pl.solve(t(sig)).items()}
        if none.any():
            with pytest.raises(N.SgError) as e:
                pl.sync()
            assert e.value.status == N.SG_ERR_NONFINITE
        else:
            pl.sync()
    for k, v in out.items():
        assert np.array_equal(np.isnan(v), none), k
    keep = ~none
    if keep.any():
        with np.errstate(all="ignore"):
            ref = oracle.direct(g, sig.astype(float), H_g=H.astype(float), G=1.0)
        force = np.hypot(ref["gr_g"], ref["gphi_g"])[keep]
        for k, v in out.items():
            scale = ref[k][keep] if k == "phi_g" else force
            assert np.linalg.norm((v - ref[k])[keep]) <= TOL[dtype] * np.linalg.norm(scale), k
