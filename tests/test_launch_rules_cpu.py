"""Kernels that are launched while the one before them may still run (programmatic dependent
launch): only after a kernel of the same call, and what that kernel writes is read by plain
loads.  The C ABI is built here on stand-ins for the launchers that record how they are
called, so no GPU is needed."""
import re
import subprocess

import pytest

from paper_2312_05492_gb300 import build as B

STANDINS = r'''
#include "abi.cu"
#include <cstdio>
#include <vector>
static std::vector<int> early_of;  // per launch: whether it may start early
static cudaError_t rec(bool early) { early_of.push_back(early); return cudaSuccess; }
namespace gi {
cudaError_t launch_prologue(const PrologueItem *, int, cudaStream_t) { return rec(false); }
cudaError_t launch_row_compress(const CompressArgs &, bool e, cudaStream_t) { return rec(e); }
cudaError_t launch_plane_compress(const CompressArgs &, bool e, cudaStream_t) { return rec(e); }
cudaError_t launch_row_decompress(const DecompressArgs &, bool e, cudaStream_t) { return rec(e); }
cudaError_t launch_plane_decompress(const DecompressArgs &, bool e, cudaStream_t) { return rec(e); }
cudaError_t launch_compress_tiles(const CompressArgs *, int, bool e, cudaStream_t, const TileSchedule *) { return rec(e); }
cudaError_t launch_decompress_tiles(const DecompressArgs *, int, bool e, cudaStream_t, const TileSchedule *) { return rec(e); }
cudaError_t launch_outlier_compaction(const CompactItem *, int, bool e, cudaStream_t) { return rec(e); }
cudaError_t launch_outlier_scatter(const ScatterItem *, int, cudaStream_t) { return rec(false); }
cudaError_t launch_histogram(const uint16_t *, uint64_t, int, uint32_t *, cudaStream_t) { return rec(false); }
cudaError_t launch_range(const float *, Dims, double, interp_config, double, interp_header *, void *, unsigned int *, int, cudaStream_t, float *) { return rec(false); }
cudaError_t launch_profile(const float *, Dims, interp_header *, int, cudaStream_t, int) { return rec(false); }
cudaError_t launch_quality(const uint32_t *, int, const float *, const float *, uint64_t, interp_quality *, void *, cudaStream_t) { return rec(false); }
cudaError_t launch_huffman_encode(const uint16_t *, unsigned long long, const uint8_t *, const uint32_t *, int, uint32_t *, uint32_t *, unsigned long long, void *, cudaStream_t) { return rec(false); }
cudaError_t launch_huffman_decode(const uint32_t *, const uint32_t *, unsigned long long, const uint8_t *, const uint32_t *, int, uint16_t *, void *, unsigned int *, cudaStream_t) { return rec(false); }
bool small_call(unsigned long long points) { return points <= 1000000ull; }
size_t range_partials_bytes() { return 1024; }
size_t quality_workspace_bytes() { return 1024; }
size_t bitmap_words_tiled(Dims d) { return (size_t)d.nz * d.ny * d.nx; }
bool huffman_codebook(const uint32_t *, int, int, uint8_t *, uint32_t *) { return true; }
unsigned long long huffman_chunks(unsigned long long n) { return n / 1024 + 1; }
unsigned long long huffman_capacity_words(unsigned long long n, int) { return n; }
size_t huffman_decode_workspace(int) { return 1024; }
size_t huffman_encode_workspace(unsigned long long) { return 1024; }
int huffman_max_len() { return 24; }
int range_blocks() { return 1; }
int sm_count() { return 152; }
}
static void show(const char *what)
{
    std::printf("%s", what);
    for (int e : early_of) std::printf(" %d", e);
    std::printf("\n");
    early_of.clear();
}
int main()
{
    alignas(16) static unsigned char p[64];  // never read: stands for every device pointer
    interp_header *h = (interp_header *)p;
    float *f = (float *)p;
    uint16_t *c = (uint16_t *)p;
    uint32_t *u = (uint32_t *)p;
    const int64_t dims[3] = {8, 16, 32}, large[3] = {128, 128, 128};
    for (int ndim = 1; ndim <= 3; ++ndim) {
        const char *name[4] = {"", "1d", "2d", "3d"};
        if (interp_decompress_nd(ndim, dims, h, f, c, u, f, 8, f, nullptr)) return 1;
        show((std::string(name[ndim]) + " list").c_str());
        if (interp_decompress_nd(ndim, dims, h, f, c, nullptr, nullptr, 0, f, nullptr)) return 1;
        show((std::string(name[ndim]) + " nolist").c_str());
        if (interp_decompress_nd(ndim, large, h, f, c, u, f, 8, f, nullptr)) return 1;
        show((std::string(name[ndim]) + " large").c_str());
    }
    interp_decompress_item it[2] = {{{8, 16, 32}, h, f, c, u, f, 0, f, 3}, {{8, 16, 32}, h, f, c, u, f, 0, f, 2}};
    if (interp_decompress_batched(it, 2, nullptr)) return 1;
    show("batch nolist");
    it[1].out_capacity = 4;
    if (interp_decompress_batched(it, 2, nullptr)) return 1;
    show("batch list");
    return 0;
}
'''


@pytest.fixture(scope="module")
def launches(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cu").write_text("#include <string>\n" + STANDINS)
    r = subprocess.run([B.nvcc(), *B.common_flags(), str(d / "rules.cu"), "-o", str(d / "rules")], capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(d / "rules")], capture_output=True, text=True)
    assert out.returncode == 0
    return {" ".join(w for w in line.split() if not w.isdigit()): [int(w) for w in line.split() if w.isdigit()]
            for line in out.stdout.splitlines()}


def test_first_kernel_of_a_call_is_never_early(launches):
    assert len(launches) == 11
    for what, early in launches.items():
        assert early[0] == 0, what


def test_small_calls_start_the_tiles_early(launches):
    for g in ("1d", "2d", "3d"):
        assert launches[g + " list"] == [0, 1]
        assert launches[g + " large"] == [0, 0]
    assert launches["batch list"] == [0, 1, 1]


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


def test_shared_memory_limits_do_not_depend_on_the_call():
    """A limit set to one call's size could be lowered by another thread's call before the
    first has launched: kernels' limits are set in one place, to sizes known at compile time."""
    for name in ("tiles.cu", "nd1.cu", "nd2.cu", "huffman.cu", "outliers.cu", "profile.cu", "quality.cu"):
        text = _source(name)
        assert "MaxDynamicSharedMemorySize" not in text, name
        for most in re.findall(r"allow_smem\([^,]+,\s*(.+?)\);", text, re.S):
            assert not re.search(r"\b(radius|nsym|n|threads|bins)\b", most), (name, most)
    for name, function in (("nd1.cu", "launch_rows"), ("nd2.cu", "launch_planes")):
        calls = re.findall(r"return " + function + r"\((.+?)\);", _source(name), re.S)
        assert len(calls) == 3
        for c in calls:
            assert "radius" not in c.split(",")[-3], c  # the limit; then early and the stream
