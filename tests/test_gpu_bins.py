"""The histogram's central bin, filled from bins at addresses of every alignment and in
numbers that are no multiple of four."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2312_05492_gb300 import fields
from paper_2312_05492_gb300 import ginterp as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


@pytest.mark.parametrize("ndim", [1, 2, 3])
@pytest.mark.parametrize("radius", [2, 3, 5, 511, 512, 513, 4097, 32767])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_central_bin(ndim, radius, shift):
    """shift: bins that the histogram starts after a 16-byte boundary."""
    x = fields.shocks((12, 40, 70), 4).cuda()
    cfg = G.Config(radius=radius, ndim=ndim)
    bufs = G.allocate(tuple(x.shape), cfg, x.device, capacity=x.numel())
    room = torch.full((2 * radius + 8,), -1, dtype=torch.int32, device="cuda")
    bufs["hist"] = room[shift:shift + 2 * radius]
    ws = torch.empty(G.interp_workspace_bytes(tuple(x.shape), cfg.to_c()), dtype=torch.uint8, device="cuda")
    G.compress_into(x, 1e-4, cfg, bufs, ws)
    torch.cuda.synchronize()
    codes = bufs["codes"].cpu().numpy().view(np.uint16)
    assert np.array_equal(bufs["hist"].cpu().numpy().view(np.uint32), O.histogram(codes, radius))
    assert bool((room[:shift] == -1).all()) and bool((room[shift + 2 * radius:] == -1).all())
