"""A kernel's walk over its work items ends, and visits each item once, when their number is
close to 2^32 (1-D fields whose rows are one point): the kernels' own stepping rule, run on
the host."""
import subprocess

import pytest

from paper_2312_05492_gb300 import build as B

PROGRAM = r'''
#include "common.cuh"
#include <cstdio>
#include <cstdlib>
// n items, `step` walkers: the items that walkers 0, 1, .. of them (the first and the last) visit
int main(int argc, char **argv)
{
    const unsigned long long n = strtoull(argv[1], nullptr, 10);
    const uint32_t step = (uint32_t)strtoul(argv[2], nullptr, 10);
    for (uint32_t first : {0u, 1u, step / 2, step - 1}) {
        unsigned long long visited = 0;
        uint32_t s = first;
        for (uint32_t next; s < (uint32_t)n; s = next) {
            if (s != first + visited * step) return 1;  // in 64 bits
            next = gi::next_item(s, step, (uint32_t)n);
            if (++visited > n) return 2;
        }
        const unsigned long long want = first < n ? (n - first + step - 1) / step : 0;
        if (visited != want) return 3;
    }
    return 0;
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("steps")
    (d / "steps.cu").write_text(PROGRAM)
    r = subprocess.run([B.nvcc(), *B.common_flags(), str(d / "steps.cu"), "-o", str(d / "steps")], capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "steps")


@pytest.mark.parametrize("n", [1, 7, 3040, 3041, 100000, 2**31, 2**32 - 3041, 2**32 - 3040, 2**32 - 2, 2**32 - 1])
@pytest.mark.parametrize("step", [1000, 3040, 3648])
def test_walk_ends(program, n, step):
    assert subprocess.run([program, str(n), str(step)], timeout=60).returncode == 0


def test_series_kernels_step_by_the_rule():
    with open(f"{B.CSRC}/nd1.cu") as f:
        text = f.read()
    assert text.count("next_item(s, step, segs)") == 2 and "s += step" not in text
