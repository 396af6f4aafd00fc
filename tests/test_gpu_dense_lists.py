"""The outlier list of fields most of whose points are outliers: blocks of 65536 points above
and below the share from which they are written word by word, rows that end inside a bitmap
word, a last block that is not whole, lists that end inside a dense block, every geometry,
against the oracle bit for bit."""
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


@pytest.mark.parametrize("ndim,shape", [(3, (33, 50, 96)), (3, (40, 41, 99)), (3, (17, 33, 260)), (2, (2, 300, 301)),
                                        (2, (1, 513, 256)), (1, (2, 40, 2049)), (1, (1, 3, 65536))])
@pytest.mark.parametrize("share", [0.15, 0.2, 0.27, 0.29, 0.6, 1.0])
@pytest.mark.parametrize("room", [1.0, 0.4])
def test_dense_blocks(ndim, shape, share, room):
    """Noise in that share of the rows' lengths (contiguous in the list), zeros elsewhere."""
    rng = np.random.default_rng(shape[2] + int(100 * share))
    x = np.zeros(shape, np.float32)
    flat = x.reshape(-1)
    block = 65536
    for b in range(0, flat.size, block):  # the first `share` of every block of points
        k = min(int(share * block), flat.size - b)
        flat[b:b + k] = rng.standard_normal(k)
    _, _, h, _ = assert_parity(x, 1e-5, G.Config(radius=8, ndim=ndim), capacity=max(1, int(room * share * x.size)))
    assert h.n_outliers > 0.7 * share * x.size
