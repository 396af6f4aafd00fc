"""The schedules that the batch tuner times: every run with the kernel's occupancy limit and
one and two CTAs per SM fewer, whatever that limit is.  The tuner is built here on stand-ins
for the kernels, so no GPU is needed."""
import subprocess

import pytest

from paper_2312_05492_gb300 import build as B

PROGRAM = r'''
#include "tune.cu"
#include <cstdlib>
namespace gi {
cudaError_t compress_tile_ctas(const CompressArgs *, int, int &) { return cudaSuccess; }
cudaError_t decompress_tile_ctas(int &) { return cudaSuccess; }
}
int interp_compress_batched_scheduled(const interp_compress_item *, int, const interp_tile_schedule *, interp_stream_t) { return 0; }
int interp_decompress_batched_scheduled(const interp_decompress_item *, int, const interp_tile_schedule *, interp_stream_t) { return 0; }
int main(int, char **argv)
{
    interp_compress_item it{};
    it.dims[0] = 73;
    for (const auto &s : candidates(&it, 1, atoi(argv[1]))) std::printf("%d %d\n", s.run, s.ctas_per_sm);
    return 0;
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("tune")
    (d / "t.cu").write_text(PROGRAM)
    r = subprocess.run([B.nvcc(), *B.common_flags(), str(d / "t.cu"), "-o", str(d / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "t")


@pytest.mark.parametrize("limit,fewer", [(6, [5, 4]), (5, [4, 3]), (2, [1]), (1, [])])
def test_candidates_follow_the_occupancy(program, limit, fewer):
    out = subprocess.run([program, str(limit)], capture_output=True, text=True, check=True).stdout
    got = [tuple(map(int, line.split())) for line in out.splitlines()]
    runs = [0, 1, 2, 4, 8, 9]  # 73 planes: nine slabs
    assert sorted(got) == sorted((r, c) for r in runs for c in [0] + fewer)
