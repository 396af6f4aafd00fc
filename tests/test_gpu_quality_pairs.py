"""The quality report's error sums (pairs of floats flushed into doubles) against numpy
float64: magnitudes inside and outside the range whose squares the pairs hold exactly,
cancelling differences, non-finite points, lengths around the vector and flush steps and
unaligned fields.

Tolerance: every addend is exact to 2^-46 of itself and the running sums are doubles, so
n <= 2^17 addends of one sign differ from numpy's sum by at most 2^-46 + 2 n 2^-53 < 4e-11
relative, in the worst order; 4e-11 it is.  Maxima and the range are exact."""
import ctypes

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


def _report(x, xr):
    hist = torch.tensor([0, 5, 9, 2], dtype=torch.int32, device="cuda")
    out = torch.zeros(ctypes.sizeof(G.interp_quality), dtype=torch.uint8, device="cuda")
    ws = torch.empty(G.interp_quality_workspace_bytes(), dtype=torch.uint8, device="cuda")
    rc = G.interp_quality_report(hist.data_ptr(), 2, x.data_ptr(), xr.data_ptr(), x.numel(), out.data_ptr(),
                                 ws.data_ptr(), ws.numel(), torch.cuda.current_stream().cuda_stream)
    assert rc == G.INTERP_OK
    return G.interp_quality.from_buffer_copy(out.cpu().numpy().tobytes())


@pytest.mark.parametrize("n", [1, 3, 4, 5, 511, 2048, 4099, 100003])
@pytest.mark.parametrize("scale,err", [(1.0, 1e-3), (1e30, 1e27), (1e-30, 1e-33), (1e-38, 3e-39), (1.0, 1e-7), (1e20, 2e20)])
@pytest.mark.parametrize("shift", [0, 1])
def test_error_sums(n, scale, err, shift):
    rng = np.random.default_rng(n + shift)
    x = (rng.standard_normal(n + shift) * scale).astype(np.float32)
    xr = (x.astype(np.float64) + rng.uniform(-err, err, n + shift)).astype(np.float32)
    if n > 100:
        x[shift + 7], x[shift + 50] = np.nan, np.inf
        xr[shift + 7], xr[shift + 50] = np.nan, np.inf
        xr[shift + 9] = x[shift + 9]
    q = _report(torch.from_numpy(x).cuda()[shift:], torch.from_numpy(xr).cuda()[shift:])
    x, xr = x[shift:], xr[shift:]
    fin = np.isfinite(x)
    d = x[fin].astype(np.float64) - xr[fin].astype(np.float64)
    sse = float((d * d).sum())
    assert q.n_finite == int(fin.sum())
    assert abs(q.sse - sse) <= 4e-11 * sse
    assert q.max_abs_err == float(np.abs(d).max())
    assert q.vmin == float(x[fin].min()) and q.vmax == float(x[fin].max())
    assert (q.n, q.n_outliers, q.n_nonzero, q.max_abs_q) == (16, 0, 7, 1)
