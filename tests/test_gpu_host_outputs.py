"""sg_solve_host into host memory of every kind: page-locked (the inverse rows
store into it), pageable, both in one call, and page-locked at an address the
row transforms cannot take (copies).  Each equals the device solve bit for bit
and leaves its neighbours alone."""
import pytest
import torch

from paper_2506_10812_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built(cuda_device):
    B.build()


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("kind", ["pinned", "mixed", "pinned view", "pinned odd address"])
def test_host_outputs(kind, dtype):
    from paper_2506_10812_gb300 import Plan
    nr, nphi = 64, 256
    n = nr * nphi
    dev = torch.device("cuda:0")
    gen = torch.Generator().manual_seed(11)
    sg = torch.rand((nr, nphi), generator=gen, dtype=dtype) + 0.5
    with Plan(nr, nphi, 0.2, 2.5, 0.05, dtype=dtype) as pl:
        ref = pl.solve(sg.to(dev))
        off = {"pinned view": 64, "pinned odd address": 1}.get(kind, 0)
        bufs, out = {}, {}
        for i, k in enumerate(ref):
            pinned = not (kind == "mixed" and i == 1)
            bufs[k] = torch.full((n + 128,), -7.0, dtype=dtype, pin_memory=pinned)
            out[k] = bufs[k][off:off + n].view(nr, nphi)
        for _ in range(2):
            pl.solve_host(sg.pin_memory(), out=out)
        pl.sync()
        for k in ref:
            assert torch.equal(out[k], ref[k].cpu()), k
            assert torch.all(bufs[k][:off] == -7.0) and torch.all(bufs[k][off + n:] == -7.0), k
