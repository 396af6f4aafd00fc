// Canonical Huffman coding of the quant-codes: the lossless stage that follows
// the histogram (Sec. V-A: the codebook is built on the host from the histogram,
// the codes are encoded and decoded on the GPU).
//
// Stream format: the codes are cut into chunks of 1024 consecutive codes; a
// chunk's codewords are concatenated most-significant bit first into 32-bit
// words (its first bit is bit 31 of its first word) and padded with zero bits
// to a whole word; offsets[k] is chunk k's first word, offsets[nchunks] the
// total.  Chunks start on word boundaries, so they decode independently.
//
// Encoding: one pass.  A tile is ENC_WARPS chunks, one warp per chunk, each lane 32
// consecutive codes; persistent CTAs take tiles in ascending order from a counter.  A
// tile sums its chunks' words, publishes the sum, puts its codewords at their bit offsets
// (a warp scan) into a shared-memory copy of the chunks, and only then looks back over
// its predecessors' published sums for the words before it (the tiles it waits for were
// taken earlier, so they run or are done), and writes its words out coalesced.  The codes
// are read once; as sizes, scan and write passes they were read twice.
// Decoding: one thread per chunk, reading its words in order.  The next 12 bits index a
// lookup table with the whole codewords they contain (up to five symbols, as bytes of 256
// around the central code R, and the bits they take); other codewords take the canonical
// rule (per length, the first codeword and the first symbol index).  Every thread does
// DEC_STEPS lookups a round whatever they yield, so the lanes of a warp stay together;
// what a round yields is appended to the thread's buffer in shared memory, whose full
// groups of 16 codes it stores itself (32 bytes: whole sectors).
#include <algorithm>
#include <cstring>
#include <queue>
#include <vector>

#include "tma.cuh"

namespace gi {
namespace {


constexpr int HCHUNK = 1024;          // codes per chunk
constexpr int HLANE = HCHUNK / 32;    // codes per lane
constexpr int ENC_WARPS = 16;         // chunks per tile
constexpr int ENC_THREADS = 32 * ENC_WARPS;
constexpr int ENC_SMEM_SYMS = 16384;  // symbols of a codebook kept in shared memory
constexpr int MAX_LEN = 24;           // longest codeword the library builds
constexpr int LUT_BITS = 12;          // lookup window: its table (32 KB) leaves two CTAs an SM
constexpr int LUT_SYMS = 5;           // symbols of an entry
constexpr uint32_t ENC_POLLS = 1u << 22;  // bounded wait for a predecessor
constexpr int TAB_THREADS = 1024;
constexpr int DEC_STEPS = 4;    // lookups a round: at most 20 codes onto at most 15 pending ones
constexpr int DEC_GROUP = 16;   // codes a thread stores at a time
constexpr int DEC_PITCH = 80;   // bytes of a thread's code buffer (35 codes and the 4 that a last entry
                                // may overwrite) and of its ring of stream words; an odd number of
                                // 16-byte units: a warp's accesses spread over the banks
constexpr int DEC_RING = 16;    // words of the ring, four 16-byte blocks
constexpr int SYM_SMEM = 4096;  // canonical symbol list kept in shared memory up to this many symbols
constexpr int DEC_THREADS = 448;  // two CTAs fit an SM, with SYM_SMEM symbols too (480, which fit with
                                  // 2800, decode 512^3 codes no faster: 247 us, 248)
static_assert(2 * (DEC_GROUP - 1 + DEC_STEPS * LUT_SYMS + LUT_SYMS - 1) <= DEC_PITCH, "a round fits the buffer");
static_assert(4 * DEC_RING <= DEC_PITCH && 31 + DEC_STEPS * MAX_LEN < 32 * 4, "a round takes at most 3 words");

// Canonical decode tables, built per call from the code lengths.
struct DecodeTables {
    uint32_t first[MAX_LEN + 2];      // first codeword of each length (canonical)
    uint32_t count[MAX_LEN + 2];      // codewords of each length
    uint32_t base[MAX_LEN + 2];       // index in `symbols` of each length's first symbol
    int max_len;
};
// followed, at TABLES_BYTES, by uint16_t symbols[2R] in canonical order
constexpr size_t TABLES_BYTES = 8512;
static_assert(sizeof(DecodeTables) <= TABLES_BYTES, "decode tables fit their room");

// A lane's 32 consecutive codes (64 bytes) as four 16-byte loads when the chunk is
// whole and the codes array is 16-byte aligned; c[j] is code j of the lane.
__device__ __forceinline__ int lane_codes(const uint16_t *__restrict__ codes, unsigned long long n,
                                          unsigned long long i0, bool vec, uint32_t w[16])
{
    if (vec && i0 + HLANE <= n) {
        const uint4 *p = reinterpret_cast<const uint4 *>(codes + i0);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint4 v = __ldg(p + k);
            w[4 * k] = v.x;
            w[4 * k + 1] = v.y;
            w[4 * k + 2] = v.z;
            w[4 * k + 3] = v.w;
        }
        return HLANE;
    }
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const unsigned long long i = i0 + 2 * k;
        const uint32_t lo = i < n ? codes[i] : 0u, hi = i + 1 < n ? codes[i + 1] : 0u;
        w[k] = lo | (hi << 16);
        cnt += (i < n) + (i + 1 < n);
    }
    return cnt;
}

__device__ __forceinline__ uint32_t code_at(const uint32_t w[16], int j) { return (w[j >> 1] >> (16 * (j & 1))) & 0xffffu; }

// ---- encode
constexpr int MAX_WORDS = (HCHUNK * MAX_LEN + 31) / 32;  // words of a chunk at the longest codewords
constexpr unsigned long long TILE_SUM = 1ull << 32, TILE_PREFIX = 2ull << 32;  // status of a tile: its own
// words, or those of all tiles up to it (low 32 bits); 0 = not published yet

__device__ __forceinline__ unsigned long long load_status(const unsigned long long *p)
{
    return *reinterpret_cast<const volatile unsigned long long *>(p);
}
__device__ __forceinline__ void publish(unsigned long long *p, unsigned long long v)
{
    *reinterpret_cast<volatile unsigned long long *>(p) = v;
}

// Words before tile t (one warp, 32 predecessors a step; looking at 320 at once, or taking
// the next tile's number early, made the tiles wait for one another longer: 161 us against
// 184 .. 207 on 2^27 codes).  A predecessor that does not publish in time sets the flag and
// gives 0: the stream is then invalid, as its flag says.
__device__ __forceinline__ uint32_t words_before(const unsigned long long *status, uint32_t t, unsigned int *bad)
{
    const int lane = threadIdx.x & 31;
    uint32_t sum = 0;
    for (long long top = (long long)t - 1;; top -= 32) {
        const long long k = top - lane;
        unsigned long long v = k >= 0 ? load_status(status + k) : TILE_PREFIX;
        uint32_t polls = 0;
        while (!__all_sync(0xffffffffu, v != 0ull)) {
            if (++polls == ENC_POLLS) {
                if (lane == 0) atomicOr(bad, 1u);
                return 0u;
            }
            if (k >= 0) v = load_status(status + k);
        }
        const uint32_t prefix = __ballot_sync(0xffffffffu, v >= TILE_PREFIX);
        const int last = prefix ? __ffs(prefix) - 1 : 31;  // the nearest tile whose prefix is known
        sum += __reduce_add_sync(0xffffffffu, lane <= last ? (uint32_t)v : 0u);
        if (prefix) return sum;
    }
}

// A lane's codewords, appended MSB first.  Words wholly inside the lane's range are
// stored, the first and the last (shared with the neighbouring lanes) are OR-ed in.
struct BitRun {
    uint32_t hi, lo;         // a 64-bit shift register: its low nacc bits are pending, bits above them are stale
    uint32_t nacc, wi, first;
    uint32_t *sw;
    uint32_t head;  // the first word, once it is full
    __device__ __forceinline__ void push(uint32_t bits, uint32_t len)  // len <= 32
    {
        hi = __funnelshift_lc(lo, hi, len);
        lo = __funnelshift_lc(0u, lo, len) | bits;
        nacc += len;
        const bool full = nacc >= 32;
        nacc &= 31u;
        const uint32_t word = __funnelshift_r(lo, hi, nacc);
        head = full && wi == first ? word : head;
        if (full && wi != first) sw[wi] = word;
        wi += full ? 1u : 0u;
    }
};

// SMEM_TAB: the codebook (length << 24 | codeword) in shared memory; otherwise a code's entry
// is put together from global memory.
template <bool SMEM_TAB>
__global__ void __launch_bounds__(ENC_THREADS, 2) k_huff_encode(const uint16_t *__restrict__ codes, unsigned long long n,
                                                               const uint8_t *__restrict__ lengths,
                                                               const uint32_t *__restrict__ codewords, int nsym,
                                                               bool vec, unsigned long long *status,
                                                               unsigned int *ticket, uint32_t tiles,
                                                               uint32_t *offsets, uint32_t *words, uint32_t nchunks,
                                                               unsigned long long capacity_words, unsigned int *bad)
{
    extern __shared__ __align__(16) uint32_t enc_sm[];  // ENC_WARPS chunk stages, then the table
    __shared__ uint32_t warp_words[ENC_WARPS];
    __shared__ uint32_t tile_s, base_s;
    uint32_t *tab = enc_sm + ENC_WARPS * MAX_WORDS;
    bool longest16 = true, packed = true;
    {
        int l16 = 0, l24 = 0;
        for (int i = threadIdx.x; i < nsym; i += ENC_THREADS) {
            const uint32_t len = lengths[i];
            l16 |= len > 16;
            l24 |= len > MAX_LEN;  // not a codebook this library builds: read unpacked
            if (SMEM_TAB) tab[i] = (len << 24) | codewords[i];
        }
        longest16 = !__syncthreads_or(l16);
        if (__syncthreads_or(l24)) packed = false;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *sw = enc_sm + warp * MAX_WORDS;
    for (;;) {
        if (threadIdx.x == 0) tile_s = atomicAdd(ticket, 1u);
        __syncthreads();  // also: every warp is done with the previous tile's shared words
        const uint32_t t = tile_s;
        if (t >= tiles) break;
        const uint32_t chunk = t * ENC_WARPS + warp;
        const unsigned long long i0 = (unsigned long long)chunk * HCHUNK + (unsigned)(lane * HLANE);
        uint32_t e[HLANE];  // table entries
        uint32_t bits = 0;
        {
            uint32_t w[16];
            // past the last chunk the lane holds no codes (its first index is past n)
            const int cnt = lane_codes(codes, n, i0, vec, w);
            if (packed) {
#pragma unroll
                for (int j = 0; j < HLANE; ++j) {
                    const uint32_t c = code_at(w, j);
                    e[j] = SMEM_TAB ? tab[c] : ((uint32_t)__ldg(lengths + c) << 24) | __ldg(codewords + c);
                }
                if (cnt < HLANE)
#pragma unroll
                    for (int j = 0; j < HLANE; ++j) e[j] = j < cnt ? e[j] : 0u;
#pragma unroll
                for (int j = 0; j < HLANE; ++j) bits = __dp4a(e[j], 0x01000000u, bits);  // the top byte
            } else {
#pragma unroll
                for (int j = 0; j < HLANE; ++j)
                    if (j < cnt) bits += lengths[code_at(w, j)];
            }
        }
        uint32_t pos = bits;  // inclusive, then exclusive scan of the lanes' bit counts
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, pos, off);
            if (lane >= off) pos += y;
        }
        const uint32_t nw = (__shfl_sync(0xffffffffu, pos, 31) + 31) / 32;  // the chunk's words
        pos -= bits;
        if (lane == 0) warp_words[warp] = nw;
        __syncthreads();
        const uint32_t v = lane < ENC_WARPS ? warp_words[lane] : 0u;
        if (warp == 0) {
            const uint32_t total = __reduce_add_sync(0xffffffffu, v);
            if (lane == 0) {
                publish(status + t, (t == 0 ? TILE_PREFIX : TILE_SUM) | total);
            }
        }
        const bool fits = nw <= (uint32_t)MAX_WORDS;  // false: lengths above MAX_LEN
        if (fits) {
            for (uint32_t i = lane; i < nw; i += 32) sw[i] = 0u;
            __syncwarp();
            BitRun r;
            r.hi = r.lo = 0;
            r.nacc = pos & 31;  // the leading part of the first word is zero
            r.wi = r.first = pos >> 5;
            r.sw = sw;
            r.head = 0;
            if (packed && longest16) {  // two codewords at a time: at most 32 bits
#pragma unroll
                for (int j = 0; j < HLANE; j += 2) {
                    const uint32_t lb = e[j + 1] >> 24;
                    r.push(((e[j] & 0xffffffu) << lb) | (e[j + 1] & 0xffffffu), (e[j] >> 24) + lb);
                }
            } else if (packed) {
#pragma unroll
                for (int j = 0; j < HLANE; ++j) r.push(e[j] & 0xffffffu, e[j] >> 24);
            } else {
#pragma unroll 1
                for (unsigned long long i = i0; i < n && i < i0 + HLANE; ++i) r.push(codewords[codes[i]], lengths[codes[i]]);
            }
            if (r.wi != r.first) atomicOr(&sw[r.first], r.head);
            if (r.nacc) atomicOr(&sw[r.wi], r.lo << (32 - r.nacc));
        }
        if (warp == 0) {
            const uint32_t b = t ? words_before(status, t, bad) : 0u;
            const uint32_t total = __reduce_add_sync(0xffffffffu, v);
            if (lane == 0) {
                if (t) publish(status + t, TILE_PREFIX | (unsigned long long)(uint32_t)(b + total));
                base_s = b;
            }
        }
        __syncthreads();
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? v : 0u);  // words of the tile before this chunk
        if (chunk < nchunks) {
            const unsigned long long w0 = (unsigned long long)base_s + before;
            if (lane == 0) {
                offsets[chunk] = (uint32_t)w0;
                if (chunk == nchunks - 1) offsets[nchunks] = (uint32_t)(w0 + nw);
            }
            if (!fits || w0 + nw > capacity_words) {  // too little room
                if (lane == 0) atomicOr(bad, 1u);
            } else {
                for (uint32_t i = lane; i < nw; i += 32) words[w0 + i] = sw[i];
            }
        }
    }
}

// ---- decode tables from the lengths (one CTA)
__global__ void __launch_bounds__(TAB_THREADS) k_huff_tables(const uint8_t *__restrict__ lengths,
                                                             const uint32_t *__restrict__ codewords, int nsym,
                                                             DecodeTables *t, uint16_t *symbols, unsigned int *bad)
{
    wait_for_previous();
    constexpr int NL = MAX_LEN + 2, NW = TAB_THREADS / 32;
    __shared__ uint32_t cnt_s[NL], base_s[NL], run_s[NL];
    __shared__ uint32_t wcnt[NW][NL];  // per warp: symbols of each length, then their offset in the length's run
    __shared__ int maxl_s;
    __shared__ unsigned int bad_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < NL) {
        cnt_s[tid] = 0u;
        run_s[tid] = 0u;
        t->first[tid] = 0xffffffffu;
    }
    if (tid == 0) {
        maxl_s = 0;
        bad_s = 0u;
    }
    __syncthreads();
    // codewords per length
    for (int s = tid; s < nsym; s += TAB_THREADS) {
        const int l = lengths[s];
        if (l > MAX_LEN) {  // not a codebook this library builds
            bad_s = 1u;
        } else if (l) {
            atomicAdd(&cnt_s[l], 1u);
            atomicMax(&maxl_s, l);
        }
    }
    __syncthreads();
    if (tid == 0) {
        uint32_t b = 0;
        for (int l = 0; l < NL; ++l) {
            base_s[l] = b;
            t->count[l] = cnt_s[l];
            t->base[l] = b;
            b += cnt_s[l];
        }
        t->max_len = maxl_s;
        *bad = bad_s;
    }
    __syncthreads();
    // canonical order: by length, ascending symbols within a length; TAB_THREADS symbols
    // at a time, ranked inside each warp, then across the warps, then after earlier rounds
    for (int s0 = 0; s0 < nsym; s0 += TAB_THREADS) {
        for (int i = tid; i < NW * NL; i += TAB_THREADS) (&wcnt[0][0])[i] = 0u;
        __syncthreads();
        const int s = s0 + tid;
        int l = s < nsym ? lengths[s] : 0;
        if (l > MAX_LEN) l = 0;
        const unsigned peers = __match_any_sync(0xffffffffu, l);
        const int rank = __popc(peers & ((1u << lane) - 1u));
        if (rank == 0) wcnt[warp][l] = (uint32_t)__popc(peers);
        __syncthreads();
        if (tid > 0 && tid < NL) {  // one thread per length: exclusive scan over the warps
            uint32_t acc = run_s[tid];
            for (int w = 0; w < NW; ++w) {
                const uint32_t c = wcnt[w][tid];
                wcnt[w][tid] = acc;
                acc += c;
            }
            run_s[tid] = acc;
        }
        __syncthreads();
        if (l) {
            const uint32_t idx = base_s[l] + wcnt[warp][l] + (uint32_t)rank;
            symbols[idx] = (uint16_t)s;
            if (idx == base_s[l]) t->first[l] = codewords[s];
        }
        __syncthreads();
    }
}

// ---- decode: one thread per chunk

// The lengths above LUT_BITS that have codewords, for the canonical rule.
struct LongCodes {
    uint4 l[MAX_LEN - LUT_BITS];  // 32 - length, first codeword, number of codewords, first symbol's index
    int n;
};

// One group of DEC_GROUP codes from shared to global memory.  VEC: bytes the destination is
// aligned to (32, 16 or 2).
template <int VEC>
__device__ __forceinline__ void store_group(uint16_t *dst, const unsigned char *src)
{
    const uint4 a = reinterpret_cast<const uint4 *>(src)[0], b = reinterpret_cast<const uint4 *>(src)[1];
    const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    if (VEC == 32) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(dst), "r"(w[0]), "r"(w[1]),
                     "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                     : "memory");
    } else if (VEC == 16) {
        reinterpret_cast<uint4 *>(dst)[0] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4 *>(dst)[1] = make_uint4(w[4], w[5], w[6], w[7]);
    } else {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            dst[2 * k] = (uint16_t)(w[k] & 0xffffu);
            dst[2 * k + 1] = (uint16_t)(w[k] >> 16);
        }
    }
}

// tg, symbols: written by the kernel before, which may still run when this one starts (no
// __restrict__: see wait_for_previous).
template <int VEC>
__global__ void __launch_bounds__(DEC_THREADS, 2) k_huff_decode(const uint32_t *__restrict__ words,
                                                               const uint32_t *__restrict__ offsets,
                                                               unsigned long long n, const DecodeTables *tg,
                                                               const uint16_t *symbols, int nsym, int nsym_smem,
                                                               uint16_t *codes, unsigned long long nchunks,
                                                               unsigned per, unsigned int *bad)
{
    wait_for_previous();
    __shared__ DecodeTables t;
    __shared__ LongCodes lc;
    __shared__ uint32_t taken;  // symbols of all entries of the lookup table
    extern __shared__ __align__(16) unsigned char dec_sm[];
    uint2 *lut = reinterpret_cast<uint2 *>(dec_sm);
    unsigned char *bufs = dec_sm + sizeof(uint2) * (1 << LUT_BITS);
    unsigned char *buf = bufs + DEC_PITCH * threadIdx.x;
    uint32_t *ring = reinterpret_cast<uint32_t *>(bufs + DEC_PITCH * (DEC_THREADS + threadIdx.x));
    uint16_t *sym_s = reinterpret_cast<uint16_t *>(bufs + 2 * DEC_PITCH * DEC_THREADS);
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(tg);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&t);
        for (int i = threadIdx.x; i < (int)(sizeof(DecodeTables) / 4); i += DEC_THREADS) dst[i] = src[i];
        for (int i = threadIdx.x; i < nsym_smem; i += DEC_THREADS) sym_s[i] = symbols[i];
    }
    __syncthreads();
    const uint16_t *sym_tab = nsym_smem ? sym_s : symbols;
    const int maxl = t.max_len;
    // symbols are bytes from here on in the lookup table: 128 on either side of R
    const int base = max(nsym / 2 - 128, 0);
    if (threadIdx.x == 0) {
        lc.n = 0;
        for (int l = LUT_BITS + 1; l <= maxl; ++l)
            if (t.count[l]) lc.l[lc.n++] = make_uint4(32u - l, t.first[l], t.count[l], t.base[l]);
    }
    // one-codeword table (symbol << 8 | length, 0: longer than the window) in the buffers' room
    uint32_t *lut1 = reinterpret_cast<uint32_t *>(bufs);
    for (int v = threadIdx.x; v < (1 << LUT_BITS); v += DEC_THREADS) {
        uint32_t e = 0;
        for (int l = 1; l <= min(maxl, LUT_BITS); ++l) {
            const uint32_t c = (uint32_t)v >> (LUT_BITS - l);
            if (c >= t.first[l] && c - t.first[l] < t.count[l]) {
                e = ((uint32_t)sym_tab[t.base[l] + (c - t.first[l])] << 8) | (uint32_t)l;
                break;
            }
        }
        lut1[v] = e;
    }
    __syncthreads();
    if (threadIdx.x == 0) taken = 0u;
    __syncthreads();
    // lookup table: word x and the low byte of y the symbols - base, then the bits taken by all
    // of them (y bits 8-11) and their number (y bits 12-14).  Number 0 and some bits: one
    // codeword whose symbol (word x) is no byte from base; number 0 and no bits: a longer codeword.
    uint32_t symbols_here = 0;
    for (int v = threadIdx.x; v < (1 << LUT_BITS); v += DEC_THREADS) {
        unsigned long long e = 0;
        uint32_t used = 0, k = 0;
        while (k < (uint32_t)LUT_SYMS) {
            const uint32_t e1 = lut1[((uint32_t)v << used) & ((1u << LUT_BITS) - 1u)];  // then zeros
            const uint32_t len = e1 & 0xffu;
            const int delta = (int)(e1 >> 8) - base;
            if (!e1 || used + len > (uint32_t)LUT_BITS) break;  // not a whole codeword of the window
            if (delta < 0 || delta > 255) {
                if (k == 0) {
                    e = e1 >> 8;
                    used = len;
                }
                break;
            }
            e |= (unsigned long long)delta << (8 * k);
            used += len;
            ++k;
        }
        lut[v] = make_uint2((uint32_t)e, (uint32_t)(e >> 32) | (used << 8) | (k << 12));
        symbols_here += k;
    }
    atomicAdd(&taken, symbols_here);
    __syncthreads();
    // A stream's bits are close to random, so this is what a lookup yields on average.  Wide
    // codes: an entry's symbols past its number are not stored (a warp's stores meet in the
    // banks: 2^27 codes of 7 bits 461 -> 319 us); narrow ones: all five are, in two whole words
    // and a half, the rest to be overwritten by the next (2.6 bits: 174 us by halves, 150; by
    // tested halves 168, and 262 against 248 where chunks differ).
    const bool wide = taken < 5u << (LUT_BITS - 1);  // 2.5 symbols

    const unsigned long long chunk = (unsigned long long)blockIdx.x * per + threadIdx.x;
    const bool live = threadIdx.x < per && chunk < nchunks;
    // The chunk's words arrive in 16-byte blocks through the ring, asynchronously and two
    // rounds ahead.  Word q counts from the block that holds the chunk's first word; words
    // before rbeg or from rend on are not the chunk's (past its end it reads zeros).
    const unsigned long long total = offsets[nchunks];
    const uint32_t off = live ? offsets[chunk] : 0u;
    const uint32_t rbeg = (uint32_t)((reinterpret_cast<uintptr_t>(words + off) >> 2) & 3u);
    const uint32_t rend = live ? rbeg + (offsets[chunk + 1] - off) : 0u;
    const uint32_t *block0 = words + off - rbeg;  // 16-byte aligned; may lie before `words`
    const long long first_ok = -(long long)off + rbeg, last_ok = (long long)(total - off) + rbeg;  // words of the stream
    uint32_t fetched = 0, rd = rbeg;
    auto fetch = [&]() {  // the next block, if the chunk has it and the ring has room
        if (fetched < rend && fetched - rd + 4 <= (uint32_t)DEC_RING) {
            uint32_t *slot = ring + (fetched & (DEC_RING - 1));
            if ((long long)fetched >= first_ok && (long long)fetched + 4 <= last_ok) {
                cp_async16(slot, block0 + fetched);
            } else {  // a block that reaches out of the stream
                for (int i = 0; i < 4; ++i) {
                    const long long q = (long long)fetched + i;
                    slot[i] = q >= first_ok && q < last_ok ? __ldg(block0 + q) : 0u;
                }
            }
            fetched += 4;
        }
        cp_async_commit();
    };
    auto take = [&]() {  // the next word
        const uint32_t v = ring[rd & (DEC_RING - 1)];
        const uint32_t r = rd < rend ? v : 0u;
        ++rd;
        return r;
    };
    for (int b = 0; b < DEC_RING / 4; ++b) fetch();
    cp_async_wait_all();
    // the next 64 bits and more: bit o of w0 is the next one
    uint32_t w0 = take(), w1 = take(), o = 0;
    int left = live ? (int)min((unsigned long long)HCHUNK, n - chunk * HCHUNK) : 0;  // codes not yet stored
    uint16_t *dst = codes + chunk * HCHUNK;
    int have = 0;         // codes in the buffer
    const uint32_t base2 = (uint32_t)base | ((uint32_t)base << 16);
    while (!__all_sync(0xffffffffu, left == 0)) {
        fetch();
        cp_async_wait_pending<2>();  // what was asked for two rounds ago is there: 5 words or more
#pragma unroll
        for (int it = 0; it < DEC_STEPS; ++it) {
            const uint32_t top = __funnelshift_l(w1, w0, o);
            const uint2 e = lut[top >> (32 - LUT_BITS)];
            uint16_t *row = reinterpret_cast<uint16_t *>(buf) + have;
            uint32_t len = (e.y >> 8) & 0xfu, k = e.y >> 12;
            // bytes to halves, plus base (no sum leaves its half)
            const uint32_t s01 = __byte_perm(e.x, 0, 0x4140) + base2, s23 = __byte_perm(e.x, 0, 0x4342) + base2;
            const uint32_t s4 = (e.y & 0xffu) + (uint32_t)base;
            if (!wide) {
                // two whole words and the half before or after them
                const uint32_t odd = (uint32_t)have & 1u;
                uint32_t *pair = reinterpret_cast<uint32_t *>(row + odd);
                pair[0] = __funnelshift_r(s01, s23, 16 * odd);
                pair[1] = __funnelshift_r(s23, s4, 16 * odd);
                row[odd ? 0 : 4] = (uint16_t)(odd ? s01 : s4);
            } else {
                row[0] = (uint16_t)s01;
                if (k > 1) row[1] = (uint16_t)(s01 >> 16);
                if (k > 2) row[2] = (uint16_t)s23;
                if (k > 3) row[3] = (uint16_t)(s23 >> 16);
                if (k > 4) row[4] = (uint16_t)s4;
            }
            if (k == 0) {
                uint32_t sym = e.x;
                if (len == 0) {  // longer than the window: the canonical rule, length by length
#pragma unroll 1
                    for (int i = 0; i < lc.n; ++i) {
                        const uint4 L = lc.l[i];
                        const uint32_t c = top >> L.x;
                        if (c >= L.y && c - L.y < L.z) {
                            sym = sym_tab[L.w + (c - L.y)];
                            len = 32u - L.x;
                            break;
                        }
                    }
                }
                if (len) {
                    row[0] = (uint16_t)sym;
                    k = 1;
                } else if (have < left) {  // not a codeword: corrupt stream, the thread stops here
                    atomicOr(bad, 1u);
                    left = 0;
                }
            }
            have += (int)k;
            o += len;
            if (o >= 32) {
                o -= 32;
                w0 = w1;
                w1 = take();
            }
        }
        // store the full groups, keep the rest at the buffer's start
        int done = 0;
        while (have - done >= DEC_GROUP && left >= DEC_GROUP) {
            store_group<VEC>(dst, buf + 2 * done);
            dst += DEC_GROUP;
            left -= DEC_GROUP;
            done += DEC_GROUP;
        }
        if (left < DEC_GROUP && have - done >= left) {  // the chunk's last codes
            const uint16_t *src = reinterpret_cast<const uint16_t *>(buf) + done;
            for (int i = 0; i < left; ++i) dst[i] = src[i];
            left = 0;
        }
        if (left == 0) {
            have = 0;
        } else if (done) {
            const uint4 a = *reinterpret_cast<const uint4 *>(buf + 2 * done), b = *reinterpret_cast<const uint4 *>(buf + 2 * done + 16);
            reinterpret_cast<uint4 *>(buf)[0] = a;
            reinterpret_cast<uint4 *>(buf)[1] = b;
            have -= done;
        }
    }
}

}  // namespace

unsigned long long huffman_chunks(unsigned long long n) { return (n + HCHUNK - 1) / HCHUNK; }

unsigned long long huffman_capacity_words(unsigned long long n, int max_len)
{
    return huffman_chunks(n) * (unsigned long long)((HCHUNK * max_len + 31) / 32);
}

size_t huffman_decode_workspace(int nsym) { return TABLES_BYTES + sizeof(uint16_t) * (size_t)nsym + 16; }

int huffman_max_len() { return MAX_LEN; }

// Host: code lengths by Huffman's construction (ties by weight, then creation
// order: symbols by index, merged nodes after) limited to max_len (lengths above
// it are cut to max_len, then the longest codewords below it are lengthened until
// the Kraft sum is at most 1), and canonical codewords.
bool huffman_codebook(const uint32_t *hist, int nsym, int max_len, uint8_t *lengths, uint32_t *codewords)
{
    if (max_len < 1 || max_len > MAX_LEN) return false;
    std::vector<int> used;
    for (int s = 0; s < nsym; ++s) {
        lengths[s] = 0;
        codewords[s] = 0;
        if (hist[s]) used.push_back(s);
    }
    if (used.empty()) return true;
    if (used.size() > (size_t(1) << max_len)) return false;  // no prefix code of max_len bits holds them
    std::vector<int> len(nsym, 0);
    if (used.size() == 1) {
        len[used[0]] = 1;
    } else {
        // nodes: leaves 0..nsym-1 (by symbol), internal nodes nsym.. in creation order
        std::vector<int> parent(2 * nsym, -1);
        using Item = std::pair<unsigned long long, int>;  // (weight, node id): smallest first
        std::priority_queue<Item, std::vector<Item>, std::greater<Item>> pq;
        for (int s : used) pq.push({hist[s], s});
        int next = nsym;
        while (pq.size() > 1) {
            const Item a = pq.top();
            pq.pop();
            const Item b = pq.top();
            pq.pop();
            parent[a.second] = next;
            parent[b.second] = next;
            pq.push({a.first + b.first, next});
            ++next;
        }
        for (int s : used) {
            int d = 0;
            for (int v = s; parent[v] >= 0; v = parent[v]) ++d;
            len[s] = d;
        }
    }
    // length limit
    int longest = 0;
    for (int s : used) longest = std::max(longest, len[s]);
    if (longest > max_len) {
        unsigned long long kraft = 0;  // in units of 2^-max_len
        for (int s : used) {
            len[s] = std::min(len[s], max_len);
            kraft += 1ull << (max_len - len[s]);
        }
        while (kraft > (1ull << max_len)) {
            int pick = -1;
            for (int s : used) {
                if (len[s] >= max_len) continue;
                if (pick < 0 || len[s] > len[pick] || (len[s] == len[pick] && hist[s] < hist[pick]) ||
                    (len[s] == len[pick] && hist[s] == hist[pick] && s > pick))
                    pick = s;
            }
            kraft -= 1ull << (max_len - len[pick] - 1);
            ++len[pick];
        }
    }
    // canonical codewords: by (length, symbol)
    std::vector<std::pair<int, int>> order;
    for (int s : used) order.push_back({len[s], s});
    std::sort(order.begin(), order.end());
    uint32_t code = 0;
    int prev = order.front().first;
    for (const auto &p : order) {
        code <<= (p.first - prev);
        codewords[p.second] = code;
        lengths[p.second] = (uint8_t)p.first;
        ++code;
        prev = p.first;
    }
    return true;
}

// A status word (8 bytes) per tile of 16 chunks; the size is stated as 4 bytes per 8
// chunks, rounded up to 256 bytes, which always holds them.  The words start after the
// first 256 bytes, or 4 bytes earlier when the workspace is only 4-byte aligned (the first
// 256 bytes hold the flag and, from 128 on, the tile counter).
size_t huffman_encode_workspace(unsigned long long n)
{
    const unsigned long long blocks = (huffman_chunks(n) + 7) / 8;
    return ((4 * blocks + 255) / 256) * 256;
}
static_assert(ENC_WARPS == 16, "status words fit huffman_encode_workspace");

template <bool SMEM_TAB>
static cudaError_t launch_encode(const uint16_t *codes, unsigned long long n, const uint8_t *lengths,
                                 const uint32_t *codewords, int nsym, uint32_t *offsets, uint32_t *words,
                                 unsigned long long capacity_words, unsigned char *ws, cudaStream_t s)
{
    const unsigned long long nch = huffman_chunks(n), tiles = (nch + ENC_WARPS - 1) / ENC_WARPS;
    const size_t smem = sizeof(uint32_t) * (ENC_WARPS * MAX_WORDS + (SMEM_TAB ? (size_t)nsym : 0));
    cudaError_t e =
        allow_smem(k_huff_encode<SMEM_TAB>, sizeof(uint32_t) * (ENC_WARPS * MAX_WORDS + (SMEM_TAB ? ENC_SMEM_SYMS : 0)));
    // flag and tile counter (the first 256 bytes) and the status words start at zero
    if (e == cudaSuccess) e = cudaMemsetAsync(ws, 0, 256 + 8 * tiles, s);
    if (e != cudaSuccess) return e;
    const bool vec = (reinterpret_cast<uintptr_t>(codes) & 15u) == 0;
    const unsigned long long wave = 2ull * sm_count();
    auto *status = reinterpret_cast<unsigned long long *>(reinterpret_cast<uintptr_t>(ws + 256) & ~(uintptr_t)7);
    k_huff_encode<SMEM_TAB><<<(unsigned)std::min(tiles, wave), ENC_THREADS, smem, s>>>(
        codes, n, lengths, codewords, nsym, vec, status, reinterpret_cast<unsigned int *>(ws + 128), (uint32_t)tiles,
        offsets, words, (uint32_t)nch, capacity_words, reinterpret_cast<unsigned int *>(ws));
    return cudaGetLastError();
}

// ws: the call's workspace (its first word is the flag).
cudaError_t launch_huffman_encode(const uint16_t *codes, unsigned long long n, const uint8_t *lengths,
                                  const uint32_t *codewords, int nsym, uint32_t *offsets, uint32_t *words,
                                  unsigned long long capacity_words, void *ws, cudaStream_t s)
{
    unsigned char *w = static_cast<unsigned char *>(ws);
    if (n == 0) {
        const cudaError_t e = cudaMemsetAsync(w, 0, sizeof(unsigned int), s);
        return e == cudaSuccess ? cudaMemsetAsync(offsets, 0, sizeof(uint32_t), s) : e;
    }
    // the codebook sits in shared memory up to ENC_SMEM_SYMS symbols (64 KB), beyond that it
    // is read through the cache
    if (nsym <= ENC_SMEM_SYMS)
        return launch_encode<true>(codes, n, lengths, codewords, nsym, offsets, words, capacity_words, w, s);
    return launch_encode<false>(codes, n, lengths, codewords, nsym, offsets, words, capacity_words, w, s);
}

// Shared memory of a decoding CTA: the lookup table, a code buffer and a ring per thread, the symbols.
static constexpr size_t decode_smem(int symbols)
{
    return sizeof(uint2) * (1 << LUT_BITS) + 2 * (size_t)DEC_PITCH * DEC_THREADS + sizeof(uint16_t) * (size_t)symbols;
}
static_assert(2 * (decode_smem(SYM_SMEM) + 1024 + 1024) <= 228 * 1024, "two decoding CTAs fit an SM");

template <int VEC>
static cudaError_t launch_decode(unsigned grid, unsigned per, cudaStream_t s, const uint32_t *words,
                                 const uint32_t *offsets, unsigned long long n, const DecodeTables *t,
                                 const uint16_t *symbols, int nsym, uint16_t *codes, unsigned long long nch,
                                 unsigned int *bad)
{
    const int nsym_smem = nsym <= SYM_SMEM ? nsym : 0;
    const cudaError_t e = allow_smem(k_huff_decode<VEC>, decode_smem(SYM_SMEM));
    if (e != cudaSuccess) return e;
    // the tables kernel is one CTA
    return launch_after(true, k_huff_decode<VEC>, grid, DEC_THREADS, decode_smem(nsym_smem), s, words, offsets, n, t,
                        symbols, nsym, nsym_smem, codes, nch, per, bad);
}

cudaError_t launch_huffman_decode(const uint32_t *words, const uint32_t *offsets, unsigned long long n,
                                  const uint8_t *lengths, const uint32_t *codewords, int nsym, uint16_t *codes,
                                  void *ws, unsigned int *bad, cudaStream_t s)
{
    DecodeTables *t = static_cast<DecodeTables *>(ws);
    uint16_t *symbols = reinterpret_cast<uint16_t *>(static_cast<unsigned char *>(ws) + TABLES_BYTES);
    k_huff_tables<<<1, TAB_THREADS, 0, s>>>(lengths, codewords, nsym, t, symbols, bad);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const unsigned long long nch = huffman_chunks(n);
    if (nch == 0) return cudaSuccess;
    // few chunks spread over the SMs, a warp of them a CTA or more; all of its threads build the table
    const unsigned long long share = (nch + 2ull * sm_count() - 1) / (2ull * sm_count());
    const unsigned per = (unsigned)std::min<unsigned long long>(DEC_THREADS, (share + 31) / 32 * 32);
    const unsigned grid = (unsigned)((nch + per - 1) / per);
    const uintptr_t a = reinterpret_cast<uintptr_t>(codes);
    if ((a & 31u) == 0) return launch_decode<32>(grid, per, s, words, offsets, n, t, symbols, nsym, codes, nch, bad);
    if ((a & 15u) == 0) return launch_decode<16>(grid, per, s, words, offsets, n, t, symbols, nsym, codes, nch, bad);
    return launch_decode<2>(grid, per, s, words, offsets, n, t, symbols, nsym, codes, nch, bad);
}

}  // namespace gi
