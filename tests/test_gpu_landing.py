"""Compression works on the values where they landed: fields that a tensor map describes and
fields that it cannot (rows or an address that are not 16-byte aligned) in one launch, runs of
one slab and of several, against the oracle bit for bit."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2312_05492_gb300 import fields
from paper_2312_05492_gb300 import ginterp as G

from _parity import assert_parity, bits

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


@pytest.mark.parametrize("offset", [0, 1, 2])
@pytest.mark.parametrize("order", [(0, 1, 2), (2, 1, 0)])
def test_landed_in_place(offset, order):
    shapes = [(9, 17, 33), (73, 16, 32), (8, 40, 68), (25, 33, 36)]
    xs, ref = [], []
    for i, shape in enumerate(shapes):
        x = fields.shocks(shape, 3 + i).numpy()
        flat = torch.empty(x.size + 4, device="cuda")
        view = flat[offset if i % 2 else 0:][:x.size].view(shape)
        view.copy_(torch.from_numpy(x))
        xs.append(view)
        ref.append(x)
    cfg = G.Config(dim_order=order, level_kind=(1, 1, 0), cubic_kind=(1, 0, 0), radius=32)
    b = G.Batch(xs, [1e-4] * len(xs), [cfg] * len(xs), capacities=[x.numel() for x in xs])
    b.round_trip()
    torch.cuda.synchronize()
    for x, cf, xr in zip(ref, b.fields, b.outs):
        eb_abs, e, twoe, inv2e = O.bounds_for(x, 1e-4, cfg.eb_mode)
        oc = O.compress(x, O.Config(order=order, level_kind=(1, 1, 0), cubic_kind=(1, 0, 0), radius=32), e, twoe,
                        inv2e, eb_abs)
        k = int(cf.host_header(refresh=True).n_outliers)
        assert k == oc.n_outliers > 0
        assert np.array_equal(cf.codes.cpu().numpy().view(np.uint16).reshape(x.shape), oc.codes)
        assert np.array_equal(bits(cf.anchors.cpu().numpy()), bits(oc.anchors))
        assert np.array_equal(cf.out_idx[:k].cpu().numpy().view(np.uint32), oc.out_idx[:k])
        assert np.array_equal(bits(cf.out_val[:k].cpu().numpy()), bits(oc.out_val[:k]))
        assert np.array_equal(cf.hist.cpu().numpy().view(np.uint32), O.histogram(oc.codes, cfg.radius))
        assert np.array_equal(bits(xr.cpu().numpy()), bits(oc.xrec))


@pytest.mark.parametrize("shape", [(10, 48, 1288), (9, 16, 32), (26, 35, 72), (17, 33, 32)])
@pytest.mark.parametrize("eb", [1e-5, 1e-6])
def test_outlier_words_of_whole_columns(shape, eb):
    """Columns inside the field with outliers in most rows: words, counts (a block of words
    that ends between a warp's rows: 41 words a row) and the list they give."""
    x = fields.shocks(shape, 5).numpy()
    _, _, h, _ = assert_parity(x, eb, G.Config(dim_order=(1, 0, 2), radius=64))
    assert h.n_outliers > x.size // 64
