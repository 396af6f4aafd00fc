"""Calls of several threads, each on its own stream, whose kernels need different amounts of
shared memory (radii, numbers of symbols): none fails, and each result is the one that the
call gives alone."""
import threading

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


@pytest.mark.parametrize("ndim,shape", [(1, (1, 3, 3000)), (2, (2, 40, 200))])
def test_radii(ndim, shape):
    x = torch.from_numpy(np.random.default_rng(5).standard_normal(shape).astype(np.float32).cumsum(axis=2)).cuda()
    cfgs = [G.Config(radius=r, ndim=ndim) for r in (4, 600, 4096)]
    # a list that holds every point: room that no call has to grow
    want = [G.compress(x, 1e-4, c, capacity=x.numel()).codes.clone() for c in cfgs]
    lengths_of = [G.huffman_codebook(torch.bincount(w.int() & 0xFFFF, minlength=2 * c.radius).int(), c.radius)
                  for w, c in zip(want, cfgs)]
    torch.cuda.synchronize()
    failed = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                ws = G.Workspace()
                for _ in range(200):
                    cf = G.compress(x, 1e-4, cfgs[i], capacity=x.numel(), workspace=ws, grow_on_overflow=False)
                    hs = G.huffman_encode(cf.codes, cfgs[i].radius, *lengths_of[i])
                    codes = G.huffman_decode(hs)
                torch.cuda.current_stream().synchronize()
                if not (torch.equal(cf.codes, want[i]) and torch.equal(codes, want[i])):
                    failed.append(f"radius {cfgs[i].radius}: other codes")
        except Exception as e:  # noqa: BLE001 - a thread's failure is the test's
            failed.append(f"radius {cfgs[i].radius}: {e}")

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(cfgs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
