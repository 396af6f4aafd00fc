"""The one-pass encoder around its tiles (16 chunks of 1024 codes): lengths around a chunk
and a tile, more tiles than one look-back step covers, codewords up to 12 bits (placed two
at a time) and up to 24 bits, against the oracle's stream word for word."""
import numpy as np
import pytest
import torch

from oracle import huffman as H
from paper_2312_05492_gb300 import ginterp as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


@pytest.mark.parametrize("n", [1, 33, 1023, 1024, 1025, 16383, 16384, 16385, 33 * 16384 + 77, 40 * 16384])
@pytest.mark.parametrize("longest", [12, 24])
def test_encoder_tiles(n, longest):
    R = 32
    # Fibonacci weights: lengths 1 .. 25 before the limit
    hist = np.zeros(2 * R, np.uint32)
    a, b = 1, 1
    for s in range(26):
        hist[3 + 2 * s if 3 + 2 * s < 2 * R else s] = a
        a, b = b, a + b
    lengths, cw = G.huffman_codebook(hist, R, longest)
    assert lengths.max() == longest
    rng = np.random.default_rng(n)
    used = np.flatnonzero(lengths)
    # short codewords mostly, and runs of the longest ones
    codes = rng.choice(used, n, p=hist[used] / hist[used].sum()).astype(np.uint16)
    long = used[lengths[used] > longest - 3]
    codes[n // 3: n // 3 + 200] = rng.choice(long, codes[n // 3: n // 3 + 200].size)
    dev = torch.from_numpy(codes.view(np.int16)).cuda()
    hs = G.huffman_encode(dev, R, lengths, cw, max_len=longest)
    torch.cuda.synchronize()
    assert int(hs.flag[:4].view(torch.int32).item()) == 0
    words, offs = H.encode_chunks(codes, lengths.astype(np.int64), cw.astype(np.uint64))
    assert np.array_equal(hs.offsets.cpu().numpy().view(np.uint32), offs)
    assert np.array_equal(hs.words[:int(offs[-1])].cpu().numpy().view(np.uint32), words)
    assert torch.equal(G.huffman_decode(hs), dev)
