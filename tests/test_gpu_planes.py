"""The 2-D kernels (strips of 64 columns, runs of chunk rows down y, 8 x 4 points a lane)
at the edges of lanes, chunks, strips and runs, both axis orders, every stencil kind, rows
of every alignment, outliers, bins beyond the shared ones and no histogram, against the
oracle bit for bit."""
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


def _planes(nz, ny, nx, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((nz, ny, nx)).cumsum(axis=2).cumsum(axis=1) * 0.1
    return (x + 0.1 * rng.standard_normal((nz, ny, nx))).astype(np.float32)


@pytest.mark.parametrize("ny,nx", [(1, 65), (2, 9), (16, 64), (17, 65), (18, 66), (31, 63), (33, 129), (35, 71), (48, 128),
                                   (49, 136), (64, 200), (15, 130), (81, 257)])
@pytest.mark.parametrize("order", [(0, 1, 2), (2, 0, 1)])
@pytest.mark.parametrize("kinds,cubic", [((0, 0, 0), (0, 0, 0)), ((1, 1, 1), (0, 0, 1)), ((1, 1, 1), (0, 1, 0)),
                                         ((1, 0, 1), (0, 1, 1))])
def test_plane_edges(ny, nx, order, kinds, cubic):
    cfg = G.Config(dim_order=order, level_kind=kinds, cubic_kind=cubic, ndim=2)
    assert_parity(_planes(2, ny, nx, 100 * ny + nx), 1e-3, cfg)


@pytest.mark.parametrize("ny,nx", [(33, 129), (40, 72), (130, 67)])
@pytest.mark.parametrize("radius,hist", [(4, True), (4097, True), (32768, True), (32768, False)])
def test_plane_outliers_and_bins(ny, nx, radius, hist):
    x = _planes(3, ny, nx, ny * nx)
    x[1, ny // 3:, nx // 2:] += 1e4
    _, _, h, _ = assert_parity(x, 1e-6, G.Config(radius=radius, eb_mode="abs", ndim=2, alpha=1.3), check_hist=hist)
    assert h.n_outliers > 0


def test_plane_runs():
    """Enough chunk rows that strips are split into several runs (a run starts with its
    first row on its own)."""
    x = _planes(1, 3000, 70, 5)
    x[0, 1024] += 50.0
    assert_parity(x, 1e-4, G.Config(dim_order=(0, 2, 1), ndim=2))
