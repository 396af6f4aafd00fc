"""The launches that a compression is said to make: a field with more bitmap blocks than the
write kernel adds up by itself takes the scan's launch too."""
import re

import pytest

from paper_2312_05492_gb300 import build as B
from paper_2312_05492_gb300 import ginterp as G


def _constant(name):
    for f in ("outliers.cu", "common.cuh"):
        with open(f"{B.CSRC}/{f}") as src:
            m = re.search(rf"constexpr int {name} = (\d+);", src.read())
        if m:
            return int(m.group(1))
    raise AssertionError(name)


def test_scan_threshold_is_the_library_s():
    assert G.SCAN_WORDS == _constant("SELF_SCAN_BLOCKS") * _constant("BITMAP_BLOCK_WORDS")


@pytest.mark.parametrize("dims,launches", [((512, 512, 512), 4), ((1024, 512, 512), 4), ((1025, 512, 512), 5),
                                           ((1024, 1024, 1024), 5), ((1, 64, 1 << 21), 4), ((4096, 2049, 1), 5),
                                           ((4096, 2048, 32), 4), ((4096, 2048, 33), 5), (None, 4)])
def test_launches(dims, launches):
    assert G.launches_compress(G.Config(), dims) == launches
