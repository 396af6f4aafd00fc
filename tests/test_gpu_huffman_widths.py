"""Decoding codes of every width: streams whose lookups hold five symbols, one, or none,
symbols in and out of the 256 around R that the table holds as bytes (and R too small for
128 below it), codebooks up to the largest (in shared memory and out of it), one chunk, fewer
chunks than the CTAs have threads for and more, last groups of every length."""
import numpy as np
import pytest
import torch

from paper_2312_05492_gb300 import ginterp as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


LARGE = 11_000_017  # more chunks than 32 for each CTA of a wave

CASES = [(R, spread, n) for R in (2, 100, 127, 128, 129, 512, 2048, 2049, 8192, 8193, 32768)
         for spread in (0.3, 0.6, 1.5, 3, 8, 30, 300, 5000) for n in (999, 33 * 1024 + 5)]
CASES += [(R, spread, LARGE) for R in (128, 512, 2049, 32768) for spread in (0.6, 3, 30, 5000)]


@pytest.mark.parametrize("R,spread,n", CASES)
def test_widths(R, spread, n):
    q = np.random.default_rng(R + n).normal(0, spread, n).round().clip(-(R - 1), R - 1)
    q[n // 2] = -(R - 1)
    q[n // 3] = R - 1
    codes = (q + R).astype(np.uint16)
    if spread == 3:
        codes[:: 1001] = 0  # outliers
    lengths, cw = G.huffman_codebook(np.bincount(codes, minlength=2 * R).astype(np.uint32), R)
    dev = torch.from_numpy(codes.view(np.int16)).cuda()
    hs = G.huffman_encode(dev, R, lengths, cw)
    out = torch.full((n + 8,), -7, dtype=torch.int16, device="cuda")
    G.huffman_decode(hs, out[:n])
    torch.cuda.synchronize()
    assert int(hs.flag[:4].cpu().numpy().view(np.uint32)[0]) == 0
    assert torch.equal(out[:n], dev)
    assert bool((out[n:] == -7).all())
    # the stream's bits are the codewords': each chunk's words hold the sum of its lengths
    bits = lengths.astype(np.int64)[codes]
    words = (np.add.reduceat(bits, np.arange(0, n, 1024)) + 31) // 32
    assert np.array_equal(np.diff(hs.offsets.cpu().numpy().view(np.uint32).astype(np.int64)), words)
