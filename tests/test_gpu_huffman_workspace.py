"""The Huffman calls' workspace and output at every alignment that they take: a workspace
that is 4-byte and not 8-byte aligned, decoded codes that are 32-, 16- and 2-byte aligned."""
import numpy as np
import pytest
import torch

from paper_2312_05492_gb300 import ginterp as G

pytestmark = pytest.mark.gpu

R = 512


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


def _codes(n):
    q = np.random.default_rng(n).normal(0, 3, n).round().clip(-40, 40)
    return (q + R).astype(np.uint16)


@pytest.mark.parametrize("n", [1, 5000, 64 * 8 * 1024, 64 * 8 * 1024 + 1])
@pytest.mark.parametrize("shift", [0, 4, 8, 12])
def test_workspace_alignment(n, shift):
    """64 x 8 x 1024 codes: the status words fill the encoder's part of the workspace."""
    codes = _codes(n)
    lengths, cw = G.huffman_codebook(np.bincount(codes, minlength=2 * R).astype(np.uint32), R)
    dev = torch.from_numpy(codes.view(np.int16)).cuda()
    want = G.huffman_encode(dev, R, lengths, cw)
    bytes_ = int(G.load().interp_huffman_workspace_bytes(n, R))
    room = torch.full((bytes_ + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    got = G.huffman_encode(dev, R, lengths, cw, ws=room[16 + shift:16 + shift + bytes_])
    torch.cuda.synchronize()
    k = want.total_words()
    assert torch.equal(got.offsets, want.offsets) and torch.equal(got.words[:k], want.words[:k])
    assert torch.equal(G.huffman_decode(got), dev)
    torch.cuda.synchronize()
    assert int(got.flag[:4].cpu().numpy().view(np.uint32)[0]) == 0
    edges = torch.cat([room[:16 + shift], room[16 + shift + bytes_:]])
    assert bool((edges == 0xA5).all())


@pytest.mark.parametrize("n", [1, 15, 16, 1024, 1025, 70001])
@pytest.mark.parametrize("shift", [0, 8, 16, 1])
def test_output_alignment(n, shift):
    codes = _codes(n)
    lengths, cw = G.huffman_codebook(np.bincount(codes, minlength=2 * R).astype(np.uint32), R)
    dev = torch.from_numpy(codes.view(np.int16)).cuda()
    hs = G.huffman_encode(dev, R, lengths, cw)
    room = torch.full((n + 64,), -7, dtype=torch.int16, device="cuda")
    G.huffman_decode(hs, room[16 + shift:16 + shift + n])
    torch.cuda.synchronize()
    assert torch.equal(room[16 + shift:16 + shift + n], dev)
    assert bool((room[:16 + shift] == -7).all()) and bool((room[16 + shift + n:] == -7).all())
