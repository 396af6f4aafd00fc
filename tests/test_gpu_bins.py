"""Histograms of many bins: codes on both sides of the bins that the 1-D and 2-D kernels keep
in shared memory when there are more than fit (2048 around R), the central bin filled from
bins at addresses of every alignment and in numbers that are no multiple of four."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2312_05492_gb300 import fields
from paper_2312_05492_gb300 import ginterp as G

from _parity import assert_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


@pytest.mark.parametrize("ndim,shape", [(1, (2, 7, 3000)), (1, (1, 600, 128)), (2, (2, 100, 150)), (2, (1, 33, 1000))])
@pytest.mark.parametrize("radius", [4096, 4097, 5001, 32768])
@pytest.mark.parametrize("spread", [30, 900, 3000])
def test_bins_around_the_window(ndim, shape, radius, spread):
    """Noise whose codes spread over +-3 `spread`: inside the 1024 on either side of R, across
    their ends, and mostly outside."""
    x = np.random.default_rng(radius + spread).standard_normal(shape).astype(np.float32)
    cfg = G.Config(radius=radius, eb_mode="abs", ndim=ndim, alpha=1.0)
    _, _, _, oc = assert_parity(x, 0.5 / spread, cfg)
    q = np.abs(oc.codes.astype(np.int64) - radius)[oc.codes != 0]
    if spread == 900:
        assert np.isin([1022, 1023, 1024, 1025], q).sum() >= 2


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
