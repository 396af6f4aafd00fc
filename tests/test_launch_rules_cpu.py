"""Kernels that are launched while the one before them may still run (programmatic dependent
launch) read what that kernel writes by plain loads: a load that calls it read-only may be
moved above the wait for that kernel."""
import re

import pytest

from paper_2312_05492_gb300 import build as B


def _source(name):
    with open(f"{B.CSRC}/{name}") as f:
        return f.read()


@pytest.mark.parametrize("name,function,params", [("huffman.cu", "k_huff_decode", ("tg", "symbols")),
                                                  ("outliers.cu", "outlier_write_block", ("bitmap",))])
def test_data_of_the_kernel_before_is_not_declared_read_only(name, function, params):
    head = re.search(function + r"\((.*?)\)\s*\n?\{", _source(name), re.S).group(1)
    for p in params:
        decl = next(d for d in head.split(",") if re.search(rf"\b{p}$", d.strip()))
        assert "__restrict__" not in decl, decl


def test_scattered_values_are_read_by_plain_loads():
    for name in ("tiles.cu", "nd1.cu", "nd2.cu"):
        assert not re.search(r"__ld\w+\([^;]*xrec", _source(name)), name
