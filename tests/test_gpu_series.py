"""The 1-D kernels (two 512-point chunks a warp, 32 points a lane) at the edges of lanes,
chunks and segments, every stencil kind, rows of every alignment, outliers, bins beyond
the shared ones and no histogram, against the oracle bit for bit."""
import numpy as np
import pytest
import torch

from paper_2312_05492_gb300 import ginterp as G

from _parity import assert_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


def _rows(nz, ny, nx, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal((nz, ny, nx)).cumsum(axis=2) + 0.1 * rng.standard_normal((nz, ny, nx))).astype(np.float32)


@pytest.mark.parametrize("nx", [1, 2, 32, 33, 255, 511, 512, 513, 514, 545, 1000, 1023, 1024, 1025, 1026, 1057, 1536,
                                1537, 2048, 2049, 3073, 5120])
@pytest.mark.parametrize("kinds,cubic", [((0, 0, 0), 0), ((1, 1, 1), 0), ((1, 1, 1), 1), ((0, 1, 1), 1), ((1, 0, 0), 0)])
def test_series_edges(nx, kinds, cubic):
    cfg = G.Config(level_kind=kinds, cubic_kind=(0, 0, cubic), ndim=1)
    assert_parity(_rows(2, 3, nx, nx), 1e-3, cfg)


@pytest.mark.parametrize("nx", [513, 1025, 1030, 2050, 4096])
@pytest.mark.parametrize("radius,hist", [(4, True), (4097, True), (32768, True), (32768, False)])
def test_series_outliers_and_bins(nx, radius, hist):
    x = _rows(1, 5, nx, 7 * nx)
    x[0, 1, nx // 2:] += 1e4
    _, _, h, _ = assert_parity(x, 1e-6, G.Config(radius=radius, eb_mode="abs", ndim=1, alpha=1.3), check_hist=hist)
    assert h.n_outliers > 0
