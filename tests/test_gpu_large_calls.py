"""The kernels that calls take whose CTAs have more than a slab, a segment or a tile to do,
against the oracle bit for bit: 3-D compression above the size up to which the wide kernel
serves every call (aligned rows, rows without a tensor map, columns cut in x and y, batches
of both kinds, the general passes), runs of several slabs, 2-D runs of several chunk rows,
the next 1-D segment landing during the levels, and encoder CTAs on their second tile."""
import numpy as np
import pytest
import torch

import oracle as O
from oracle import huffman as H
from paper_2312_05492_gb300 import fields
from paper_2312_05492_gb300 import ginterp as G

from _parity import assert_parity, bits

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _slabs(shape):
    return ((shape[2] + 31) // 32) * ((shape[1] + 15) // 16) * max(1, (shape[0] + 6) // 8)


def _noisy(shape, seed):
    """A smooth field with steps and a little noise: outliers of the tighter bounds everywhere."""
    x = fields.shocks(shape, seed).numpy()
    return x + 1e-3 * np.random.default_rng(seed).standard_normal(shape).astype(np.float32)


WIDE_SLABS = 10  # per SM: two for each of five CTAs


@pytest.mark.parametrize("shape", [(201, 203, 235), (201, 203, 256), (201, 197, 232), (201, 208, 228), (137, 250, 310)])
@pytest.mark.parametrize("eb,order", [(1e-3, (0, 1, 2)), (2e-5, (2, 0, 1))])
def test_large_fields(shape, eb, order):
    assert _slabs(shape) > WIDE_SLABS * _sms()
    cfg = G.Config(dim_order=order, cubic_kind=(0, 1, 0), radius=64)
    _, _, h, _ = assert_parity(_noisy(shape, shape[2]), eb, cfg)
    assert (eb > 1e-4) or h.n_outliers > 1000


@pytest.mark.parametrize("cfg", [dict(domain_x=32), dict(radius=1024), dict(radius=1024, domain_x=32)])
@pytest.mark.parametrize("shape", [(201, 203, 256), (201, 203, 235)])
def test_large_fields_general_passes(shape, cfg):
    assert _slabs(shape) > WIDE_SLABS * _sms()
    assert_parity(_noisy(shape, 3), 2e-5, G.Config(dim_order=(1, 0, 2), **cfg))


def _same_as_oracle(x, cf, xr, eb, cfg):
    eb_abs, e, twoe, inv2e = O.bounds_for(x, eb, cfg.eb_mode)
    oc = O.compress(x, O.Config(order=cfg.dim_order, level_kind=cfg.level_kind, cubic_kind=cfg.cubic_kind,
                                radius=cfg.radius, domain_x=cfg.domain_x), e, twoe, inv2e, eb_abs)
    k = int(cf.host_header(refresh=True).n_outliers)
    assert k == oc.n_outliers
    assert np.array_equal(cf.codes.cpu().numpy().view(np.uint16).reshape(x.shape), oc.codes)
    assert np.array_equal(bits(cf.anchors.cpu().numpy()), bits(oc.anchors))
    assert np.array_equal(cf.out_idx[:k].cpu().numpy().view(np.uint32), oc.out_idx[:k])
    assert np.array_equal(bits(cf.out_val[:k].cpu().numpy()), bits(oc.out_val[:k]))
    assert np.array_equal(cf.hist.cpu().numpy().view(np.uint32), O.histogram(oc.codes, cfg.radius))
    assert np.array_equal(bits(xr.cpu().numpy()), bits(oc.xrec))


@pytest.mark.parametrize("domain", [8, 32])
def test_large_mixed_batch(domain):
    """Rows with and without a tensor map, of 16- and 8-byte aligned codes and of neither, in one
    launch; domain 32: one field that needs the general passes among them."""
    shapes = [(73, 203, 256), (73, 120, 235), (60, 130, 300), (49, 97, 228), (120, 160, 96)]
    assert sum(_slabs(s) for s in shapes) > WIDE_SLABS * _sms()
    xs = [_noisy(s, 10 + i) for i, s in enumerate(shapes)]
    cfgs = [G.Config(dim_order=(1, 2, 0), radius=64, domain_x=domain if i == 2 else 8) for i in range(len(xs))]
    b = G.Batch([torch.from_numpy(x).cuda() for x in xs], [2e-5] * len(xs), cfgs, capacities=[x.size for x in xs])
    b.round_trip()
    torch.cuda.synchronize()
    for x, cf, xr, cfg in zip(xs, b.fields, b.outs, cfgs):
        _same_as_oracle(x, cf, xr, 2e-5, cfg)


@pytest.mark.parametrize("run", [2, 3, 100])
@pytest.mark.parametrize("large", [False, True])
def test_runs_of_several_slabs(run, large):
    shapes = [(201, 203, 235), (73, 120, 256), (73, 131, 228)] if large else [(73, 33, 35), (40, 17, 64), (33, 18, 36)]
    xs = [_noisy(s, 20 + i) for i, s in enumerate(shapes)]
    cfg = G.Config(dim_order=(2, 1, 0), radius=64)
    b = G.Batch([torch.from_numpy(x).cuda() for x in xs], [2e-5] * len(xs), [cfg] * len(xs), capacities=[x.size for x in xs])
    b.csched = b.dsched = G.interp_tile_schedule(run, 0)
    b.round_trip()
    torch.cuda.synchronize()
    for x, cf, xr in zip(xs, b.fields, b.outs):
        _same_as_oracle(x, cf, xr, 2e-5, cfg)


def _walk(shape, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal(shape).cumsum(axis=2)
    if shape[1] > 1:
        x = x.cumsum(axis=1) * 0.1
    return (x + 0.1 * rng.standard_normal(shape)).astype(np.float32)


@pytest.mark.parametrize("shape", [(1, 16 * 700, 300), (40, 16 * 16 + 5, 643), (9, 16 * 120 + 1, 520)])
@pytest.mark.parametrize("order", [(0, 1, 2), (0, 2, 1)])
def test_planes_with_runs(shape, order):
    """More items than warps (16 a SM) if every run were one chunk row: runs of several."""
    rows, strips = (shape[1] + 15) // 16, (shape[2] + 63) // 64
    assert shape[0] * rows * strips > 16 * _sms()
    x = _walk(shape, 5)
    x[-1, shape[1] // 2] += 50.0
    _, _, h, _ = assert_parity(x, 1e-5, G.Config(dim_order=order, ndim=2, radius=64))
    assert h.n_outliers > 0


@pytest.mark.parametrize("rows,nx", [(8000, 1027), (4000, 2048), (5000, 1031)])
def test_series_with_several_segments_a_warp(rows, nx):
    """More segments of 1024 points than compression (20 a SM) and decompression (24) have warps."""
    assert rows * ((nx + 1023) // 1024) > 24 * _sms()
    x = _walk((1, rows, nx), 6)
    x[0, rows - 7, nx // 3:] += 1e3
    _, _, h, _ = assert_parity(x, 1e-5, G.Config(ndim=1, radius=64))
    assert h.n_outliers > 0


def _stream(codes, lengths, codewords, chunk=1024):
    """The oracle's encode_chunks on arrays."""
    L = lengths[codes]
    nch = -(-codes.size // chunk)
    starts = np.arange(nch) * chunk
    offs = np.concatenate([[0], np.cumsum((np.add.reduceat(L, starts) + 31) // 32)])
    before = np.cumsum(L) - L
    at = 32 * np.repeat(offs[:-1], chunk)[:codes.size] + before - np.repeat(before[starts], chunk)[:codes.size]
    bit = np.zeros(32 * offs[-1], np.uint8)
    for k in range(int(lengths.max())):  # bit k of every codeword that has one
        m = L > k
        bit[at[m] + k] = (codewords[codes[m]] >> (L[m] - 1 - k)) & 1
    return np.packbits(bit).view(">u4").astype(np.uint32), offs.astype(np.uint32)


@pytest.mark.parametrize("extra", [0, 77])
@pytest.mark.parametrize("longest", [12, 24])
def test_encoder_second_tiles(extra, longest):
    """More tiles of 16384 codes than two CTAs a SM take at first, codewords of one bit to the
    longest in every chunk."""
    n = (2 * _sms() * 2 + 5) * 16384 + extra
    R = 32
    hist = np.zeros(2 * R, np.uint32)
    a, b = 1, 1
    for s in range(26):
        hist[3 + 2 * s if 3 + 2 * s < 2 * R else s] = a
        a, b = b, a + b
    lengths, cw = G.huffman_codebook(hist, R, longest)
    used = np.flatnonzero(lengths)
    codes = np.random.default_rng(n).choice(used, n, p=hist[used] / hist[used].sum()).astype(np.uint16)
    codes[::999] = used[-1]
    dev = torch.from_numpy(codes.view(np.int16)).cuda()
    hs = G.huffman_encode(dev, R, lengths, cw, max_len=longest)
    torch.cuda.synchronize()
    assert int(hs.flag[:4].view(torch.int32).item()) == 0
    words, offs = _stream(codes, lengths.astype(np.int64), cw.astype(np.int64))
    w20, o20 = H.encode_chunks(codes[:20 * 1024], lengths.astype(np.int64), cw.astype(np.uint64))
    assert np.array_equal(offs[:21], o20) and np.array_equal(words[:o20[-1]], w20)
    assert np.array_equal(hs.offsets.cpu().numpy().view(np.uint32), offs)
    assert np.array_equal(hs.words[:int(offs[-1])].cpu().numpy().view(np.uint32), words)
    assert torch.equal(G.huffman_decode(hs), dev)
