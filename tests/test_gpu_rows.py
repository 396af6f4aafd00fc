"""Rows that are not 16-byte aligned (the landing and the write-out by one lane per
x-position): every remainder of nx by 4 and 8, rows shorter than a column, columns cut
in x and y, with and without outliers, against the oracle bit for bit."""
import numpy as np
import pytest
import torch

from paper_2312_05492_gb300 import fields
from paper_2312_05492_gb300 import ginterp as G

from _parity import assert_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


@pytest.mark.parametrize("nx", [1, 7, 31, 33, 34, 36, 38, 63, 65, 70, 97])
@pytest.mark.parametrize("nz,ny", [(9, 16), (17, 33), (26, 15)])
@pytest.mark.parametrize("eb,radius", [(1e-3, 512), (1e-5, 16)])
def test_unaligned_rows(nx, nz, ny, eb, radius):
    x = np.random.default_rng(nx * 100 + ny).standard_normal((nz, ny, nx)).astype(np.float32).cumsum(axis=0)
    x += fields.sines((nz, ny, nx), 3).numpy()
    _, _, h, _ = assert_parity(x, eb, G.Config(dim_order=(1, 2, 0), cubic_kind=(0, 1, 0), radius=radius))
    if eb == 1e-5:
        assert h.n_outliers > 0
