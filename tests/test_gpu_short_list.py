"""A field with more outliers than its list has room for: the reconstruction does not depend
on what the output buffer held, and is the oracle's with 0 in the place of the outliers that
are not listed, in every geometry, alignment and call form."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as O
from paper_2312_05492_gb300 import ginterp as G

from _parity import assert_parity, bits

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


def _noise(shape, seed):
    return np.random.default_rng(seed).standard_normal(shape).astype(np.float32)


def _expected(oc, cap):
    val = oc.out_val.copy()
    val[cap:] = 0
    return bits(O.decompress(dataclasses.replace(oc, out_val=val)))


@pytest.mark.parametrize("ndim,shape", [(3, (17, 33, 64)), (3, (9, 18, 35)), (3, (49, 49, 49)), (2, (2, 33, 72)),
                                        (2, (1, 40, 131)), (1, (1, 5, 2048)), (1, (2, 3, 1031))])
@pytest.mark.parametrize("room", [1, 100, 0.5])
def test_short_list(ndim, shape, room):
    x = _noise(shape, 7 * ndim + shape[2])
    cap = room if room >= 1 else int(room * x.size / 8)
    cf, _, h, oc = assert_parity(x, 1e-4, G.Config(radius=16, ndim=ndim), capacity=cap)
    assert h.status == G.STATUS_CAPACITY and h.n_outliers > cap
    want = _expected(oc, cap)
    for held in (float("nan"), 1e30):
        out = torch.full(shape, held, device="cuda")
        G.decompress_into(cf, out)
        assert np.array_equal(bits(out.cpu().numpy()), want)


def test_short_lists_in_a_batch():
    """Short lists beside one with room."""
    shapes = [(49, 49, 49), (33, 17, 96), (20, 40, 68), (2, 48, 64)]
    xs = [_noise(s, i) for i, s in enumerate(shapes)]
    cfgs = [G.Config(radius=16, ndim=3)] * 3 + [G.Config(radius=16, ndim=2)]
    caps = [x.size // 16 for x in xs]
    caps[1] = xs[1].size
    b = G.Batch([torch.from_numpy(x).cuda() for x in xs], [1e-4] * 4, cfgs, capacities=caps)
    got = []
    for held in (float("nan"), -3e7):
        for o in b.outs:
            o.fill_(held)
        b.round_trip()
        torch.cuda.synchronize()
        got.append([bits(o.cpu().numpy()) for o in b.outs])
    for i, (x, cfg) in enumerate(zip(xs, cfgs)):
        _, _, h, oc = assert_parity(x, 1e-4, cfg, capacity=x.size)
        assert (h.n_outliers > caps[i]) == (i != 1)
        want = _expected(oc, caps[i])
        assert np.array_equal(got[0][i], want) and np.array_equal(got[1][i], want)
