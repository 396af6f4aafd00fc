// Outlier stream compaction (Sec. V-A: outliers are gathered and stored
// losslessly), the outlier scatter of decompression, and the standalone
// quant-code histogram (Fig. 1 "histogram", Sec. V-A).
//
// Compaction is ordered: the compression kernel writes one bitmap word per
// 32 x-positions of every row and adds the popcount of each non-zero word to
// the counter of its 2048-word block.  One CTA per block of words expands its
// words into a list of indices in shared memory, then all threads write (index, value)
// pairs at consecutive addresses, their loads independent of one another (a thread
// writing its own words' pairs, or a warp taking word after word, waits for every value
// in turn: 28 us and 76 us against 8 us on eight cubes of up to 240^3 points).  Words are in ascending linear-index order, so the outlier list comes out sorted by
// index with no sort and no atomics.  A CTA's offset is the sum of the counters
// before its own, which it adds up itself while they are few (SELF_SCAN_BLOCKS);
// larger fields have a one-CTA scan turn the counts into offsets first.
#include <algorithm>
#include <cstring>

#include "common.cuh"

namespace gi {
namespace {

constexpr int SCAN_THREADS = 1024;
constexpr int WRITE_THREADS = 256;
constexpr int WRITE_WARPS = WRITE_THREADS / 32;
constexpr int WORDS_PER_THREAD = BITMAP_BLOCK_WORDS / WRITE_THREADS;  // 8
constexpr uint32_t WRITE_LIST = 6144;  // indices expanded at a time (24 KB)
// A block with more outliers (28% of its points) is written word by word, a warp a word and a
// lane a point: the list is expanded by the threads whose words it holds at a time, 24 of 256
// when every point is an outlier.  92% of 64^3 points 137 -> 38 us, of 512^3 502 -> 375 us;
// 21% of 3 x 1001 x 1003: 80 us by the list, 98 word by word; 33% of 512^3: 212 and 237.
constexpr uint32_t WRITE_DENSE = 3 * WRITE_LIST;
static_assert(WRITE_LIST == 3 * BITMAP_BLOCK_WORDS, "three values of every word of a block fit the list's room");
// up to here (a field of about 2^28 points) a CTA adds up at most 4096 counters (16 a
// thread, from L2), which costs less than the scan's launch (5 us on 512^3 points)
constexpr int SELF_SCAN_BLOCKS = 4096;

// Bin R of a histogram whose tile kernel left it out (it is the most frequent code by
// far): N minus every other bin.  All threads of a block of T threads.
template <int T>
__device__ void fill_central_bin(uint32_t *hist, int radius, unsigned long long n)
{
    __shared__ unsigned long long part[T / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // bin R, taken off at the start
    unsigned long long others = threadIdx.x == 0 ? 0ull - hist[radius] : 0ull;
    // 16-byte loads, several in flight a thread: a block reads up to 65536 bins
    const int n4 = (reinterpret_cast<uintptr_t>(hist) & 15u) == 0 ? 2 * radius / 4 : 0;
#pragma unroll 4
    for (int i = threadIdx.x; i < n4; i += T) {
        const uint4 v = reinterpret_cast<const uint4 *>(hist)[i];
        others += (unsigned long long)v.x + v.y + v.z + v.w;
    }
#pragma unroll 1
    for (int c = 4 * n4 + threadIdx.x; c < 2 * radius; c += T) others += hist[c];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) others += __shfl_xor_sync(0xffffffffu, others, off);
    __syncthreads();
    if (lane == 0) part[warp] = others;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < T / 32; ++w) t += part[w];
        hist[radius] = (uint32_t)(n - t);
    }
}

// Exclusive scan of the block counts in place; total -> header; central bin.
__device__ void outlier_scan_block(uint32_t *blockcnt, int nblk, interp_header *hdr, unsigned long long capacity,
                                   uint32_t *hist, int radius, unsigned long long n)
{
    __shared__ unsigned long long warp_sum[SCAN_THREADS / 32];
    __shared__ unsigned long long carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nblk; base += SCAN_THREADS) {
        const int i = base + threadIdx.x;
        const unsigned long long v = i < nblk ? blockcnt[i] : 0u;
        unsigned long long incl = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
        }
        if (lane == 31) warp_sum[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            unsigned long long w = warp_sum[lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, w, off);
                if (lane >= off) w += y;
            }
            warp_sum[lane] = w;  // inclusive over warps
        }
        __syncthreads();
        const unsigned long long before = carry + (warp ? warp_sum[warp - 1] : 0ull) + incl - v;
        // offsets of blocks fit in 32 bits because N < 2^32
        if (i < nblk) blockcnt[i] = (uint32_t)before;
        __syncthreads();
        if (threadIdx.x == SCAN_THREADS - 1) carry = before + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        hdr->n_outliers = carry;
        if (carry > capacity) hdr->status |= INTERP_STATUS_CAPACITY;
    }
    if (hist) fill_central_bin<SCAN_THREADS>(hist, radius, n);
}

// Block-wide room of the write kernel: the list, and the warps' counts.
__shared__ uint32_t w_list[WRITE_LIST];
__shared__ uint32_t w_sum[WRITE_WARPS];

// A thread's words (from w0 on), the outliers in them, those before them in the block, and the
// block's.
struct Words {
    uint32_t wv[WORDS_PER_THREAD];
    uint32_t pos, total;
};
__device__ __forceinline__ void load_words(Words &W, const uint32_t *bitmap, uint32_t words, uint32_t words_per_row, int ny,
                                           int nz, bool row_major, uint32_t w0)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t cnt = 0;
#pragma unroll
    for (int k = 0; k < WORDS_PER_THREAD; ++k) {
        const uint32_t w = w0 + k;
        W.wv[k] = w < words ? bitmap[row_major ? (size_t)w : tiled_word(w, words_per_row, ny, nz)] : 0u;
        cnt += __popc(W.wv[k]);
    }
    // block exclusive scan of the threads' counts
    uint32_t incl = cnt;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    if (lane == 31) w_sum[warp] = incl;
    __syncthreads();
    W.pos = incl - cnt;
    W.total = 0;
#pragma unroll
    for (int w = 0; w < WRITE_WARPS; ++w) {
        if (w < warp) W.pos += w_sum[w];
        W.total += w_sum[w];
    }
}

// The outliers of bitmap block b of a field, written from position `start` of its list on.
// bitmap: by the kernel before (no __restrict__: see wait_for_previous).
__device__ void outlier_write_block(const uint32_t *bitmap, uint32_t words, uint32_t words_per_row, int nx,
                                    int ny, int nz, const float *__restrict__ x, uint32_t *out_idx, float *out_val,
                                    unsigned long long capacity, bool row_major, uint32_t b, unsigned long long start)
{
    const uint32_t w0 = b * (uint32_t)BITMAP_BLOCK_WORDS + (uint32_t)(threadIdx.x * WORDS_PER_THREAD);
    Words W;
    load_words(W, bitmap, words, words_per_row, ny, nz, row_major, w0);
    uint32_t *list = w_list, (&wv)[WORDS_PER_THREAD] = W.wv, pos = W.pos;
    const uint32_t total = W.total;
    for (uint32_t from = 0; from < total; from += WRITE_LIST) {
        const uint32_t n = min(WRITE_LIST, total - from);
        // this thread's outliers at positions [from, from + n); their bits are cleared
#pragma unroll
        for (int k = 0; k < WORDS_PER_THREAD; ++k) {
            if (!wv[k] || pos >= from + n) continue;
            const uint32_t w = w0 + k, row = w / words_per_row;
            const uint32_t first = row * (uint32_t)nx + (w - row * words_per_row) * 32u;
            while (wv[k] && pos < from + n) {
                list[pos - from] = first + (uint32_t)(__ffs(wv[k]) - 1);
                wv[k] &= wv[k] - 1u;
                ++pos;
            }
        }
        __syncthreads();
        const unsigned long long out = start + from;
        const uint32_t room = out < capacity ? (uint32_t)min((unsigned long long)n, capacity - out) : 0u;
#pragma unroll 4
        for (uint32_t i = threadIdx.x; i < room; i += WRITE_THREADS) {
            const uint32_t idx = list[i];
            out_idx[out + i] = idx;
            out_val[out + i] = __ldg(x + idx);
        }
        __syncthreads();
    }
}

// Ordered compaction of the outliers of n fields: every field's non-empty bitmap blocks
// (after one scan block per field with many of them).
struct CompactField {
    const uint32_t *bitmap;
    uint32_t *blockcnt;
    uint32_t words, words_per_row;
    int nx, ny, nz;
    const float *x;
    uint32_t *out_idx;
    float *out_val;
    unsigned long long capacity;
    interp_header *hdr;
    int nblk;
    bool row_major;
    uint32_t *hist;  // fills bin R when not null
    int radius;
    unsigned long long n;
    int b0;          // first write block of the field
    int scanned;     // blockcnt holds offsets (k_outlier_scan), not counts
};

// outlier_write_block for a block of many outliers.  Out of line: its registers are not the list's.
__device__ __noinline__ void outlier_write_dense(const CompactField &F, uint32_t b, unsigned long long start)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t i0 = (uint32_t)(threadIdx.x * WORDS_PER_THREAD), w0 = b * (uint32_t)BITMAP_BLOCK_WORDS + i0;
    uint32_t *bits = w_list, *at = w_list + BITMAP_BLOCK_WORDS, *first = w_list + 2 * BITMAP_BLOCK_WORDS;
    Words W;
    load_words(W, F.bitmap, F.words, F.words_per_row, F.ny, F.nz, F.row_major, w0);
#pragma unroll
    for (int k = 0; k < WORDS_PER_THREAD; ++k) {
        const uint32_t w = w0 + k, row = w / F.words_per_row;
        bits[i0 + k] = W.wv[k];
        at[i0 + k] = W.pos;
        first[i0 + k] = row * (uint32_t)F.nx + (w - row * F.words_per_row) * 32u;
        W.pos += __popc(W.wv[k]);
    }
    __syncthreads();
    const uint32_t room = (uint32_t)min((unsigned long long)W.total, F.capacity - start);
    const float *__restrict__ x = F.x;
    uint32_t *out_idx = F.out_idx + start;
    float *out_val = F.out_val + start;
    constexpr int AT_ONCE = 4;  // words of a warp whose values are on their way together
    static_assert(BITMAP_BLOCK_WORDS % (AT_ONCE * WRITE_WARPS) == 0, "whole rounds");
    for (int i = warp; i < BITMAP_BLOCK_WORDS; i += AT_ONCE * WRITE_WARPS) {
        uint32_t p[AT_ONCE], idx[AT_ONCE];
        float v[AT_ONCE];
#pragma unroll
        for (int j = 0; j < AT_ONCE; ++j) {
            const uint32_t m = bits[i + j * WRITE_WARPS];
            idx[j] = first[i + j * WRITE_WARPS] + lane;
            p[j] = (m >> lane & 1u) ? at[i + j * WRITE_WARPS] + __popc(m & ((1u << lane) - 1u)) : room;
            v[j] = p[j] < room ? __ldg(x + idx[j]) : 0.0f;
        }
#pragma unroll
        for (int j = 0; j < AT_ONCE; ++j)
            if (p[j] < room) {
                out_idx[p[j]] = idx[j];
                out_val[p[j]] = v[j];
            }
    }
}

struct CompactBatch {
    CompactField f[kMaxBatch];
    int n;
};

__global__ void __launch_bounds__(SCAN_THREADS) k_outlier_scan(const __grid_constant__ CompactBatch B)
{
    wait_for_previous();
    const CompactField &F = B.f[blockIdx.x];
    if (F.scanned) outlier_scan_block(F.blockcnt, F.nblk, F.hdr, F.capacity, F.hist, F.radius, F.n);
}

__global__ void __launch_bounds__(WRITE_THREADS) k_outlier_write(const __grid_constant__ CompactBatch B)
{
    wait_for_previous();
    int fi = 0;
    while (fi + 1 < B.n && B.f[fi + 1].b0 <= (int)blockIdx.x) ++fi;
    const CompactField &F = B.f[fi];
    const int b = (int)blockIdx.x - F.b0;
    unsigned long long start;
    uint32_t own;
    if (F.scanned) {
        start = F.blockcnt[b];
        const unsigned long long end = b + 1 < F.nblk ? F.blockcnt[b + 1] : F.hdr->n_outliers;
        own = (uint32_t)(end - start);
        if (own == 0) return;
    } else {
        const bool last = b == F.nblk - 1;
        own = F.blockcnt[b];
        if (b == 0 && F.hist) fill_central_bin<WRITE_THREADS>(F.hist, F.radius, F.n);
        if (own == 0 && !last) return;
        // the counters before this block's
        __shared__ unsigned long long part[WRITE_WARPS];
        unsigned long long sum = 0;
        for (int i = threadIdx.x; i < b; i += WRITE_THREADS) sum += F.blockcnt[i];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
        __syncthreads();
        start = 0;
#pragma unroll
        for (int w = 0; w < WRITE_WARPS; ++w) start += part[w];
        if (last && threadIdx.x == 0) {
            F.hdr->n_outliers = start + own;
            if (start + own > F.capacity) F.hdr->status |= INTERP_STATUS_CAPACITY;
        }
        if (own == 0) return;
    }
    if (start >= F.capacity) return;  // beyond the caller's capacity
    if (own > WRITE_DENSE)
        outlier_write_dense(F, (uint32_t)b, start);
    else
        outlier_write_block(F.bitmap, F.words, F.words_per_row, F.nx, F.ny, F.nz, F.x, F.out_idx, F.out_val, F.capacity,
                            F.row_major, (uint32_t)b, start);
}

// Outlier values of n fields into their reconstructions: `blocks` blocks per field.
struct ScatterField {
    const interp_header *hdr;
    const uint32_t *idx;
    const float *val;
    unsigned long long capacity;
    float *xrec;
    unsigned long long points;
};

struct ScatterBatch {
    ScatterField f[kMaxBatch];
    int n, blocks;
};

__global__ void k_outlier_scatter(const __grid_constant__ ScatterBatch B)
{
    wait_for_previous();
    const ScatterField &F = B.f[blockIdx.x / B.blocks];
    const unsigned long long b = blockIdx.x % B.blocks;
    unsigned long long n = F.hdr->n_outliers;
    const unsigned long long step = (unsigned long long)B.blocks * blockDim.x;
    unsigned long long i = b * blockDim.x + threadIdx.x;
    if (n > F.capacity) {
        // a list that was too short: the outliers past its last index (it is ascending) have
        // no value, and read as 0 and not as what xrec happened to hold
        n = F.capacity;
        for (unsigned long long k = F.idx[n - 1] + 1ull + i; k < F.points; k += step) F.xrec[k] = 0.0f;
    }
    for (; i + 3 * step < n; i += 4 * step) {  // four independent pairs in flight
        uint32_t k[4];
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            k[j] = __ldcs(F.idx + i + j * step);
            v[j] = __ldcs(F.val + i + j * step);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) F.xrec[k[j]] = v[j];
    }
    for (; i < n; i += step) F.xrec[F.idx[i]] = F.val[i];
}

// Standalone histogram: per-CTA shared bins (register count for the central
// code R, which dominates for accurate predictions, Sec. V-A), flushed once.
constexpr int HIST_THREADS = 512;
constexpr int HIST_SMEM_MAX_BINS = 16384;

__global__ void __launch_bounds__(HIST_THREADS) k_histogram(const uint16_t *__restrict__ codes,
                                                            unsigned long long n, int radius, int vec,
                                                            uint32_t *hist)
{
    extern __shared__ uint32_t hs[];
    const int bins = 2 * radius;
    const bool smem = bins <= HIST_SMEM_MAX_BINS;
    if (smem)
        for (int i = threadIdx.x; i < bins; i += HIST_THREADS) hs[i] = 0u;
    __syncthreads();
    uint32_t central = 0;
    auto count = [&](uint32_t c) {
        if (c == (uint32_t)radius) {
            ++central;
        } else if (c < (uint32_t)bins) {
            if (smem) atomicAdd(&hs[c], 1u);
            else atomicAdd(&hist[c], 1u);
        }
    };
    const unsigned long long tid = (unsigned long long)blockIdx.x * HIST_THREADS + threadIdx.x;
    const unsigned long long nth = (unsigned long long)gridDim.x * HIST_THREADS;
    unsigned long long done = 0;
    if (vec) {
        const uint4 *c8 = reinterpret_cast<const uint4 *>(codes);
        const unsigned long long n8 = n / 8;
        for (unsigned long long i = tid; i < n8; i += nth) {
            const uint4 v = __ldcs(c8 + i);
            const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                count(w4[k] & 0xffffu);
                count(w4[k] >> 16);
            }
        }
        done = n8 * 8;
    }
    for (unsigned long long i = done + tid; i < n; i += nth) count(codes[i]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) central += __shfl_xor_sync(0xffffffffu, central, off);
    if ((threadIdx.x & 31) == 0 && central) {
        if (smem) atomicAdd(&hs[radius], central);
        else atomicAdd(&hist[radius], central);
    }
    if (smem) {
        __syncthreads();
        for (int i = threadIdx.x; i < bins; i += HIST_THREADS) {
            const uint32_t h = hs[i];
            if (h) atomicAdd(&hist[i], h);
        }
    }
}

}  // namespace

cudaError_t launch_outlier_compaction(const CompactItem *items, int n, bool early, cudaStream_t s)
{
    if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
    CompactBatch B;
    std::memset(&B, 0, sizeof(B));
    int blocks = 0;
    bool scan = false;
    for (int i = 0; i < n; ++i) {
        const CompactItem &it = items[i];
        CompactField &F = B.f[i];
        F.bitmap = it.bitmap;
        F.blockcnt = it.blockcnt;
        F.words = (uint32_t)it.words;  // N < 2^32
        F.words_per_row = (uint32_t)((it.d.nx + 31) / 32);
        F.nx = it.d.nx;
        F.ny = it.d.ny;
        F.nz = it.d.nz;
        F.x = it.x;
        F.out_idx = it.out_idx;
        F.out_val = it.out_val;
        F.capacity = (unsigned long long)it.capacity;
        F.hdr = it.hdr;
        F.nblk = (int)((it.words + BITMAP_BLOCK_WORDS - 1) / BITMAP_BLOCK_WORDS);
        F.row_major = it.row_major;
        F.hist = it.central_hist;
        F.radius = it.radius;
        F.n = (unsigned long long)it.d.nz * it.d.ny * it.d.nx;
        F.b0 = blocks;
        F.scanned = F.nblk > SELF_SCAN_BLOCKS;
        scan = scan || F.scanned;
        blocks += F.nblk;
    }
    B.n = n;
    if (scan) {
        const cudaError_t e = launch_after(false, k_outlier_scan, n, SCAN_THREADS, 0, s, B);
        if (e != cudaSuccess) return e;
    }
    return launch_after(early, k_outlier_write, blocks, WRITE_THREADS, 0, s, B);
}

cudaError_t launch_outlier_scatter(const ScatterItem *items, int n, cudaStream_t s)
{
    if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
    ScatterBatch B;
    std::memset(&B, 0, sizeof(B));
    for (int i = 0; i < n; ++i) B.f[i] = ScatterField{items[i].hdr, items[i].idx, items[i].val,
                                                      (unsigned long long)items[i].capacity, items[i].xrec,
                                                      (unsigned long long)items[i].points};
    B.n = n;
    // a full SM of threads (the stores are scattered), but no more than the lists may need
    uint64_t most = 1;
    for (int i = 0; i < n; ++i) most = std::max<uint64_t>(most, items[i].capacity);
    B.blocks = (int)std::min<uint64_t>(std::max(1, 8 * sm_count() / n), (most + 1023) / 1024);
    k_outlier_scatter<<<B.blocks * n, 256, 0, s>>>(B);
    return cudaGetLastError();
}

cudaError_t launch_histogram(const uint16_t *codes, uint64_t n, int radius, uint32_t *hist, cudaStream_t s)
{
    const int bins = 2 * radius;
    const size_t smem = bins <= HIST_SMEM_MAX_BINS ? sizeof(uint32_t) * (size_t)bins : 0;
    if (smem > 48 * 1024) {
        cudaError_t e = allow_smem(k_histogram, sizeof(uint32_t) * HIST_SMEM_MAX_BINS);
        if (e != cudaSuccess) return e;
    }
    const int vec = (reinterpret_cast<uintptr_t>(codes) % 16) == 0;
    unsigned long long blocks = (n + 8ull * HIST_THREADS * 8 - 1) / (8ull * HIST_THREADS * 8);
    const unsigned long long cap = 4ull * sm_count();
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    k_histogram<<<(unsigned)blocks, HIST_THREADS, smem, s>>>(codes, (unsigned long long)n, radius, vec, hist);
    return cudaGetLastError();
}

}  // namespace gi
