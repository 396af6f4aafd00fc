"""The quality report's sum of squared errors against exact integer arithmetic: no less
accurate than a sum in doubles, whose every addend is rounded to 2^-53 of itself.

Tolerance, in units of 2^-53 of the (positive) sum.  Up to 4 points: a pending sum goes into
its double in 2 roundings, and at most 2 additions of threads' sums follow; what the pending
sum itself loses is below 2^-60: 5 in all.  Up to 2^17 points: at most 2 such transfers and
2 additions a thread (15 points), then 20 additions in a block and 21 over the blocks: 64."""
import ctypes
from fractions import Fraction

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


def _sse(x, xr):
    hist = torch.tensor([0, 5, 9, 2], dtype=torch.int32, device="cuda")
    out = torch.zeros(ctypes.sizeof(G.interp_quality), dtype=torch.uint8, device="cuda")
    ws = torch.empty(G.interp_quality_workspace_bytes(), dtype=torch.uint8, device="cuda")
    rc = G.interp_quality_report(hist.data_ptr(), 2, x.data_ptr(), xr.data_ptr(), x.numel(), out.data_ptr(),
                                 ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
    assert rc == G.INTERP_OK
    return G.interp_quality.from_buffer_copy(out.cpu().numpy().tobytes()).sse


def _exact(x, xr):
    total = 0
    for a, b in zip(x.tolist(), xr.tolist()):
        d = int(Fraction(a) * 2**149) - int(Fraction(b) * 2**149)  # float32 values are multiples of 2^-149
        total += d * d
    return Fraction(total, 2**298)


@pytest.mark.parametrize("n,seeds", [(1, 12), (2, 8), (4, 8), (65, 2), (4099, 2), (100003, 1)])
@pytest.mark.parametrize("kind", ["small", "cancelling", "spread", "bins"])
@pytest.mark.parametrize("shift", [0, 1])
def test_sum_is_a_double_sum(n, seeds, kind, shift):
    units = 5 if n <= 4 else 64
    for seed in range(seeds):
        rng = np.random.default_rng(1000 * seed + n)
        x = rng.standard_normal(n + shift).astype(np.float32)
        if kind == "small":
            xr = (x + rng.uniform(-1e-3, 1e-3, n + shift)).astype(np.float32)
        elif kind == "cancelling":
            xr = rng.standard_normal(n + shift).astype(np.float32)
        elif kind == "spread":  # differences that two floats are needed for
            x = (x * 10.0 ** rng.uniform(-6, 6, n + shift)).astype(np.float32)
            xr = (x + rng.uniform(-10, 10, n + shift)).astype(np.float32)
        else:  # values far below the bound, as in a density field
            x = np.exp(3 * x).astype(np.float32)
            xr = (np.round(x / 0.2) * np.float32(0.2)).astype(np.float32)
        got = _sse(torch.from_numpy(x).cuda()[shift:], torch.from_numpy(xr).cuda()[shift:])
        want = _exact(x[shift:], xr[shift:])
        assert abs(Fraction(got) - want) <= want * units / 2**53, (seed, float(abs(Fraction(got) - want) / want) * 2**53)
