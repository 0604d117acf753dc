"""The indirect term's reduction at the edges of its decomposition (one column,
short and long rows, odd and unaligned rows, more column groups than blocks)
with zeros, denormals and both signs among the densities, and with scale-height
fields; against the oracle's kernel summed in FP64.  Tolerance 1e-12 of the sum
of the terms' magnitudes (FP64 accumulation of rounded inputs).  With a
scale-height field the factor per cell takes the plan's radii, which an FP32 plan
holds in FP32: the reference is evaluated on those."""
import numpy as np
import pytest
import torch

import oracle
from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()
    oracle.build()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nr,nphi,off,fields", [(5, 1, 0, False), (7, 3, 0, True), (33, 64, 0, False), (33, 64, 1, True),
                                                (3, 257, 0, True), (600, 24, 0, False), (2, 45000, 0, False)])
def test_reduction_edges(nr, nphi, off, fields, dtype):
    from paper_2506_10812_gb300 import Plan
    rng = np.random.default_rng(nr * 7919 + nphi)
    npdt = np.float32 if dtype == torch.float32 else np.float64
    g = oracle.Grid(nr, nphi, 0.2, 2.5)
    R, Pm = g.mesh()
    s = [rng.normal(1.0, 1.0, R.shape).astype(npdt) for _ in range(2)]
    for a in s:
        a.flat[:: 5] = 0.0
        a.flat[1:: 11] = np.finfo(npdt).tiny / 8
    H = [(R * rng.uniform(0.01, 3.0, R.shape)).astype(npdt) for _ in range(2)] if fields else [None, None]
    ref, mag = [], []
    for a, (sig, h) in enumerate(zip(s, H)):
        r = R.astype(npdt).astype(float) if fields else R
        Ha = h.astype(float) if fields else R * (0.05, 0.004)[a]
        w = np.sqrt(2) * 1.3 * g.du * g.dphi * sig.astype(float) * r * r * oracle.indirect_kernel(r / Ha, Ha)
        ref.append([np.sum(w * np.cos(Pm)), np.sum(w * np.sin(Pm))])
        mag.append(np.sum(np.abs(w) * (np.abs(np.cos(Pm)) + np.abs(np.sin(Pm)))))
    ref = np.array(ref)
    dev = torch.device("cuda:0")

    def place(a):                              # `off` elements past an aligned address
        if a is None:
            return None
        buf = torch.empty(a.size + off, dtype=dtype, device=dev)
        buf[off:] = torch.tensor(a.ravel(), dtype=dtype, device=dev)
        return buf[off:].view(nr, nphi)

    with Plan(nr, nphi, 0.2, 2.5, 0.05, 0.004, G=1.3, dtype=dtype, method="direct", H_g=place(H[0]), H_d=place(H[1])) as pl:
        x, y = place(s[0]), place(s[1])
        ab = pl.indirect(x, y)
        assert torch.equal(ab, pl.indirect(x, y))
        ab = ab.cpu().numpy()
    assert ab.shape == ref.shape
    assert np.all(np.abs(ab - ref) <= 1e-12 * np.array(mag)[:, None])
