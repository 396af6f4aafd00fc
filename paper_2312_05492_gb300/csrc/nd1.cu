// 1-D G-Interp (Sec. IV-A: 512-point chunks, anchors every 512 points, strides 256 .. 1),
// compression and decompression, in registers.
//
// A warp owns a segment of 1024 consecutive points of one row, i.e. two chunks; a lane
// holds 32 consecutive points in registers.  Strides 256 .. 32 touch only the lanes'
// first points (warp shuffles, four levels); strides 16 .. 1 stay inside a lane but for
// the nearest known points of its neighbours (three shuffles a level).  So the nine
// levels need no shared memory and no block barrier between them.  The kernels that
// this replaced ran the levels over a 2048-point tile in shared memory with a barrier
// after each; 3.4 .. 4.2 warp instructions a point and the barriers bound them.
//
// Shared memory only turns the lanes' 32-point runs into coalesced accesses: the input
// lands there (cp.async, 16 bytes where the rows allow it, issued a segment ahead) in
// runs of 36 floats (or 40 codes), so that a warp's 16-byte reads of 32 runs fall in
// distinct banks; codes and reconstructions leave through it the same way.
//
// Bound by instruction issue (about 25 a point: prediction 2 .. 9, quantization 11,
// histogram 3), then by HBM: 4N read + 2N written.
#include "lanes.cuh"

namespace gi {
namespace {

// warps per CTA (each on its own segments) and CTAs per SM: 20 warps of 96 registers for
// compression (229 us against 252 with 24 warps of 80 on 64 x 2^21 points), 24 of 80 for
// decompression (171 us against 181)
struct Shape {
    int warps, ctas;
};
constexpr Shape RC{4, 5}, RD{8, 3};
constexpr int RUN = 32;               // points per lane
constexpr int SEG = 32 * RUN;         // points per warp
constexpr int CHUNK = 512, CLANES = CHUNK / RUN;  // lanes per chunk
constexpr int LEVELS = 9;
constexpr int VP = 36;                // floats per landed run (32 and 4 of padding)
constexpr int KP = 40;                // codes per landed run
constexpr size_t R_V = sizeof(float) * 32 * VP, R_K = sizeof(uint16_t) * 32 * KP;
constexpr size_t R_LQ = 0;                       // level constants
constexpr size_t R_SPARE = R_LQ + 16 * LEVELS;   // one word per lane for updates that count nothing
constexpr size_t R_WARPS = R_SPARE + 4 * 32;     // then per warp: value runs, code runs
constexpr size_t R_WARP = R_V + R_K;
constexpr size_t R_HIST = R_WARPS + R_WARP * RC.warps;  // compression: the bins
static_assert(R_WARPS % 16 == 0 && R_HIST % 16 == 0, "shared layout alignment");

extern __shared__ __align__(128) unsigned char r_smem[];

__device__ __forceinline__ LevelQ level_of(int l)
{
    const float4 q = reinterpret_cast<const float4 *>(r_smem + R_LQ)[l];
    return LevelQ{q.x, q.y, q.z};
}

// What a lane does with the points of its segment: quantize and count (compression), or
// apply the stored codes (decompression).  v: the 32 values; cw: the 32 codes, two a word.
struct Lane {
    float v[RUN];
    uint32_t cw[RUN / 2];
};

struct Ctx : Bins {
    uint32_t cbias;
    float Rf;
    int lane, cl;          // lane, lane within its chunk
    float closing;         // the point after the segment (an anchor), in every lane
    int last;              // last in-field offset from the segment's start (SEG when it is whole)
};

// Neighbour-count rule (Sec. IV-B.1).
template <int KIND>
__device__ __forceinline__ float predict(float m3, float m1, float p1, float p3, bool hm3, bool hp1, bool hp3)
{
    float p = sp_linear(m1, p1);
    if (KIND != K_LINEAR) {
        const float ql = sp_quad_left(m3, m1, p1), qr = sp_quad_right(m1, p1, p3), cu = cubic_of<KIND>(m3, m1, p1, p3);
        p = hm3 ? (hp3 ? cu : ql) : (hp3 ? qr : p);
    }
    return hp1 ? p : m1;
}

// One point: value v (compression: the original on entry, x' on return) and its code.
template <int MODE, bool OUTL>
__device__ __forceinline__ uint32_t point(const Ctx &c, const LevelQ &q, float &v, float p, uint32_t code, bool counts)
{
    if (MODE != DECODE) {
        code = quantize(v, p, q, c.cbias, c.Rf, v);
        count<MODE>(c, code, counts);
    } else {
        const float xq = p + code_to_q(code, c.cbias) * q.twoe;
        v = OUTL && code == 0u ? v : xq;  // an outlier's stored value is there already
    }
    return code;
}

// Stride 32 T: only the lanes' first points, through shuffles.
template <int MODE, bool OUTL, bool FULL, int T, int KIND>
__device__ __forceinline__ void coarse_level(Lane &L, const Ctx &c)
{
    constexpr int l = T == 8 ? 8 : (T == 4 ? 7 : (T == 2 ? 6 : 5));
    const LevelQ q = level_of(l);
    const float a = L.v[0];
    const float m1 = __shfl_sync(0xffffffffu, a, c.lane - T), m3 = __shfl_sync(0xffffffffu, a, c.lane - 3 * T);
    float p1 = __shfl_sync(0xffffffffu, a, c.lane + T), p3 = __shfl_sync(0xffffffffu, a, c.lane + 3 * T);
    if (c.lane + T == 32) p1 = c.closing;
    if (c.lane + 3 * T == 32) p3 = c.closing;
    const bool hm3 = c.cl >= 3 * T;
    const bool hp1 = FULL || RUN * (c.lane + T) <= c.last;
    const bool hp3 = c.cl + 3 * T <= CLANES && (FULL || RUN * (c.lane + 3 * T) <= c.last);
    const float p = predict<KIND>(m3, m1, p1, p3, hm3, hp1, hp3);
    const bool mine = (c.cl & (2 * T - 1)) == T;
    float v = a;
    const uint32_t code = point<MODE, OUTL>(c, q, v, p, L.cw[0] & 0xffffu,
                                                mine && (FULL || RUN * c.lane <= c.last));
    if (mine) {
        L.v[0] = v;
        if (MODE != DECODE) L.cw[0] = code;
    }
}

// Stride S <= 16: P = 16 / S points of the lane.
template <int MODE, bool OUTL, bool FULL, int S, int KIND>
__device__ __forceinline__ void lane_level(Lane &L, const Ctx &c, float next0)
{
    constexpr int l = S == 16 ? 4 : (S == 8 ? 3 : (S == 4 ? 2 : (S == 2 ? 1 : 0)));
    constexpr int P = RUN / (2 * S);
    const LevelQ q = level_of(l);
    float before = 0.0f, after = 0.0f;  // the known points next to the lane's run
    if (KIND != K_LINEAR) {
        before = __shfl_up_sync(0xffffffffu, L.v[RUN - 2 * S], 1);
        after = __shfl_down_sync(0xffffffffu, P > 1 ? L.v[P > 1 ? 2 * S : 0] : next0, 1);
    }
    const bool first = c.cl == 0, last = c.cl == CLANES - 1;  // the run starts / ends its chunk
#pragma unroll
    for (int i = 0; i < P; ++i) {
        constexpr int D = 2 * S;
        const int o = (2 * i + 1) * S;
        const float m1 = L.v[D * i], p1 = i + 1 < P ? L.v[i + 1 < P ? D * (i + 1) : 0] : next0;
        const float m3 = i > 0 ? L.v[i > 0 ? D * (i - 1) : 0] : before;
        const float p3 = i + 2 < P ? L.v[i + 2 < P ? D * (i + 2) : 0] : (i + 2 == P ? next0 : after);
        float p;
        bool in = true;
        if (FULL) {
            if (KIND == K_LINEAR) {
                p = sp_linear(m1, p1);
            } else {
                p = cubic_of<KIND>(m3, m1, p1, p3);
                if (i == 0) p = first ? sp_quad_right(m1, p1, p3) : p;
                if (i == P - 1) p = last ? sp_quad_left(m3, m1, p1) : p;
            }
        } else {
            const int n = RUN * c.lane + o;
            in = n <= c.last;
            p = predict<KIND>(m3, m1, p1, p3, i > 0 || !first, n + S <= c.last,
                              (i < P - 1 || !last) && n + 3 * S <= c.last);
        }
        const uint32_t w = L.cw[o / 2];
        const uint32_t code =
            point<MODE, OUTL>(c, q, L.v[o], p, S == 1 ? w >> 16 : w & 0xffffu, in);
        if (MODE != DECODE) L.cw[o / 2] = S == 1 ? w + (code << 16) : code;
    }
}

template <int MODE, bool OUTL, bool FULL, int S, int KIND>
__device__ __forceinline__ void any_level(Lane &L, const Ctx &c, float next0)
{
    if constexpr (S >= RUN) coarse_level<MODE, OUTL, FULL, S / RUN, KIND>(L, c);
    else lane_level<MODE, OUTL, FULL, S, KIND>(L, c, next0);
}

template <int MODE, bool OUTL, bool FULL, int S>
__device__ __forceinline__ void levels_from(Lane &L, const Ctx &c, int kind0, int kind1, int kind2, float next0)
{
    if (S == 16) {  // the lanes' first points are final: the next lane's serves all finer strides
        next0 = __shfl_down_sync(0xffffffffu, L.v[0], 1);
        if (c.lane == 31) next0 = c.closing;
    }
    const int kind = S == 1 ? kind0 : (S == 2 ? kind1 : kind2);  // coarser levels than 4 follow stride 4
    if (kind == K_LINEAR) any_level<MODE, OUTL, FULL, S, K_LINEAR>(L, c, next0);
    else if (kind == K_NAK) any_level<MODE, OUTL, FULL, S, K_NAK>(L, c, next0);
    else any_level<MODE, OUTL, FULL, S, K_NATURAL>(L, c, next0);
    if constexpr (S > 1) levels_from<MODE, OUTL, FULL, S / 2>(L, c, kind0, kind1, kind2, next0);
}

// Kinds of the three level classes (strides 1, 2, 4 and more).
struct Kinds {
    int k0, k1, k2;
};
__device__ __forceinline__ Kinds kinds_of(const interp_header *h)
{
    const int cubic = h->cfg.cubic_kind[2] ? K_NATURAL : K_NAK;
    return Kinds{h->cfg.level_kind[0] ? cubic : K_LINEAR, h->cfg.level_kind[1] ? cubic : K_LINEAR,
                 h->cfg.level_kind[2] ? cubic : K_LINEAR};
}

// Segment `s`: its row and its first point.
struct Seg {
    unsigned long long base;  // linear index of its first point
    uint32_t row;
    int x0, valid;            // first point in the row, in-field points
};
__device__ __forceinline__ Seg seg_of(uint32_t s, uint32_t per_row, int nx)
{
    Seg g;
    g.row = s / per_row;
    g.x0 = (int)(s - g.row * per_row) * SEG;
    g.valid = min(SEG, nx - g.x0);
    g.base = (unsigned long long)g.row * (unsigned)nx + (unsigned)g.x0;
    return g;
}

// ------------------------------------------------------------ compression
__device__ __forceinline__ void land_values(float *land, const float *x, const Seg &g, bool vec, int lane)
{
    const float *src = x + g.base;
    if (vec) {
#pragma unroll
        for (int i = 0; i < RUN / 4; ++i) {
            const int e = 4 * (32 * i + lane);  // rows are whole groups of 4
            if (e < g.valid) cp_async16(land + (e >> 5) * VP + (e & 31), src + e);
        }
    } else {
#pragma unroll 8
        for (int i = 0; i < RUN; ++i)
            if (32 * i + lane < g.valid) cp_async4(land + i * VP + lane, src + 32 * i + lane);
    }
    cp_async_commit();
}

template <int MODE>
__global__ void __launch_bounds__(32 * RC.warps, RC.ctas) k_row_compress(const CompressArgs a, uint32_t per_row,
                                                                   uint32_t segs)
{
    wait_for_previous();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nx = a.dims.nx;
    const int bins = MODE == ENCODE_GBINS ? LANE_WINDOW : 2 * a.radius;  // in shared memory
    const int win0 = MODE == ENCODE_GBINS ? a.radius - LANE_WINDOW / 2 : 0;
    uint32_t *hs = reinterpret_cast<uint32_t *>(r_smem + R_HIST);
    store_levels<LEVELS>(a.hdr, reinterpret_cast<float4 *>(r_smem + R_LQ));
    for (int i = threadIdx.x; i < bins; i += 32 * RC.warps) hs[i] = 0u;
    __syncthreads();
    float *land = reinterpret_cast<float *>(r_smem + R_WARPS + R_WARP * warp);
    uint16_t *stage = reinterpret_cast<uint16_t *>(r_smem + R_WARPS + R_WARP * warp + R_V);
    const bool vec = (nx & 3) == 0 && (reinterpret_cast<uintptr_t>(a.x) & 15u) == 0;
    const bool vec_codes = (nx & 7) == 0 && (reinterpret_cast<uintptr_t>(a.codes) & 15u) == 0;
    const Kinds kd = kinds_of(a.hdr);
    const uint32_t wpr = (uint32_t)(nx + 31) / 32u, apr = (uint32_t)(nx - 1) / CHUNK + 1u;
    Ctx c;
    c.cbias = kMagicBits - (uint32_t)a.radius;
    c.R = (uint32_t)a.radius;
    c.Rf = (float)a.radius;
    c.hist = smem_u32(hs);
    c.win0 = (uint32_t)win0;
    c.spare = smem_u32(r_smem + R_SPARE) + 4u * lane;
    c.hist_g = a.hist;
    c.lane = lane;
    c.cl = lane & (CLANES - 1);

    // segments go to CTAs first, then to their warps: few segments spread over the SMs
    uint32_t s = blockIdx.x + gridDim.x * (uint32_t)warp;
    const uint32_t step = gridDim.x * RC.warps;
    float closing = 0.0f;
    if (s < segs) {
        const Seg g = seg_of(s, per_row, nx);
        land_values(land, a.x, g, vec, lane);
        if (g.x0 + SEG < nx) closing = __ldg(a.x + g.base + SEG);
    }
    for (uint32_t next; s < segs; s = next) {
        const Seg g = seg_of(s, per_row, nx);
        next = next_item(s, step, segs);
        cp_async_wait_all();
        __syncwarp();
        Lane L;
#pragma unroll
        for (int i = 0; i < RUN / 4; ++i) {
            const float4 f = reinterpret_cast<const float4 *>(land + lane * VP)[i];
            L.v[4 * i] = f.x;
            L.v[4 * i + 1] = f.y;
            L.v[4 * i + 2] = f.z;
            L.v[4 * i + 3] = f.w;
        }
        c.closing = closing;
        __syncwarp();
        if (next < segs) {  // the next segment lands during the levels
            const Seg n = seg_of(next, per_row, nx);
            land_values(land, a.x, n, vec, lane);
            if (n.x0 + SEG < nx) closing = __ldg(a.x + n.base + SEG);
        }
        const bool full = g.x0 + SEG < nx;  // both chunks and the closing point inside the row
        c.last = full ? SEG : nx - 1 - g.x0;
        L.cw[0] = c.R;  // the anchors' code
        if (full) levels_from<MODE, false, true, 256>(L, c, kd.k0, kd.k1, kd.k2, 0.0f);
        else levels_from<MODE, false, false, 256>(L, c, kd.k0, kd.k1, kd.k2, 0.0f);
        const int p0 = g.x0 + RUN * lane;  // the lane's first point in the row
        if (c.cl == 0 && p0 < nx) a.anchors[(size_t)g.row * apr + (uint32_t)p0 / CHUNK] = L.v[0];
        // outlier word of the lane's 32 points (row-major bitmap) and its block count
        uint32_t word = 0u, least = 0xffffffffu;
#pragma unroll
        for (int i = 0; i < RUN / 2; ++i) least = __vminu2(least, L.cw[i]);
        if (__any_sync(0xffffffffu, (least & 0xffffu) == 0u || least < 0x10000u)) {
#pragma unroll
            for (int i = 0; i < RUN / 2; ++i)
                word |= ((L.cw[i] & 0xffffu) == 0u ? 1u : 0u) << (2 * i) | (L.cw[i] < 0x10000u ? 2u : 0u) << (2 * i);
            const int in = nx - p0;
            if (in < RUN) word &= in > 0 ? (1u << in) - 1u : 0u;
            const unsigned long long gw = (unsigned long long)g.row * wpr + (uint32_t)p0 / 32u;
            if (word) atomicAdd(a.blockcnt + gw / BITMAP_BLOCK_WORDS, (uint32_t)__popc(word));
        }
        if (p0 < nx) a.bitmap[(unsigned long long)g.row * wpr + (uint32_t)p0 / 32u] = word;
        // codes: lane runs -> coalesced
        __syncwarp();  // the stage's previous contents are written out
#pragma unroll
        for (int i = 0; i < RUN / 8; ++i)
            reinterpret_cast<uint4 *>(stage + lane * KP)[i] =
                make_uint4(L.cw[4 * i], L.cw[4 * i + 1], L.cw[4 * i + 2], L.cw[4 * i + 3]);
        __syncwarp();
        uint16_t *dst = a.codes + g.base;
        if (vec_codes) {
#pragma unroll
            for (int i = 0; i < RUN / 8; ++i) {
                const int e = 8 * (32 * i + lane);
                if (e < g.valid)
                    *reinterpret_cast<uint4 *>(dst + e) =
                        *reinterpret_cast<const uint4 *>(stage + (e >> 5) * KP + (e & 31));
            }
        } else {
#pragma unroll 8
            for (int i = 0; i < RUN; ++i)
                if (32 * i + lane < g.valid) dst[32 * i + lane] = stage[i * KP + lane];
        }
    }
    if (a.hist) {
        __syncthreads();
        for (int i = threadIdx.x; i < bins; i += 32 * RC.warps)
            if (hs[i]) atomicAdd(&a.hist[win0 + i], hs[i]);
    }
}

// ---------------------------------------------------------- decompression
__device__ __forceinline__ void land_codes(uint16_t *land, const uint16_t *codes, const Seg &g, int width, int lane)
{
    const uint16_t *src = codes + g.base;
    if (width == 8) {
#pragma unroll
        for (int i = 0; i < RUN / 8; ++i) {
            const int e = 8 * (32 * i + lane);
            if (e < g.valid) cp_async16(land + (e >> 5) * KP + (e & 31), src + e);
        }
    } else if (width == 2) {
#pragma unroll 8
        for (int i = 0; i < RUN / 2; ++i) {
            const int e = 2 * (32 * i + lane);
            if (e < g.valid) cp_async4(land + (e >> 5) * KP + (e & 31), src + e);
        }
    } else {
#pragma unroll 8
        for (int i = 0; i < RUN; ++i)
            if (32 * i + lane < g.valid) land[i * KP + lane] = __ldg(src + 32 * i + lane);
    }
    cp_async_commit();
}

__global__ void __launch_bounds__(32 * RD.warps, RD.ctas) k_row_decompress(const DecompressArgs a, uint32_t per_row,
                                                                     uint32_t segs)
{
    wait_for_previous();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nx = a.dims.nx;
    store_levels<LEVELS>(a.hdr, reinterpret_cast<float4 *>(r_smem + R_LQ));
    __syncthreads();
    float *stage = reinterpret_cast<float *>(r_smem + R_WARPS + R_WARP * warp);
    uint16_t *land = reinterpret_cast<uint16_t *>(r_smem + R_WARPS + R_WARP * warp + R_V);
    const bool vec = (nx & 3) == 0 && (reinterpret_cast<uintptr_t>(a.xrec) & 15u) == 0;
    const uintptr_t ca = reinterpret_cast<uintptr_t>(a.codes);
    const int width = (nx & 7) == 0 && (ca & 15u) == 0 ? 8 : ((nx & 1) == 0 && (ca & 3u) == 0 ? 2 : 1);
    const Kinds kd = kinds_of(a.hdr);
    const uint32_t apr = (uint32_t)(nx - 1) / CHUNK + 1u;
    Ctx c;
    c.R = (uint32_t)a.hdr->cfg.radius;
    c.cbias = kMagicBits - c.R;
    c.Rf = 0.0f;
    c.hist = c.spare = c.win0 = 0u;
    c.hist_g = nullptr;
    c.lane = lane;
    c.cl = lane & (CLANES - 1);

    // anchors of a segment: lanes 0 and 16 (their first points), lane 31 (the closing point)
    auto anchor_of = [&](const Seg &g) {
        const int i = lane == 31 ? 2 : lane / CLANES;
        const bool need = c.cl == 0 || lane == 31;
        return need && g.x0 + CHUNK * i < nx
                   ? __ldg(a.anchors + (size_t)g.row * apr + (uint32_t)g.x0 / CHUNK + i) : 0.0f;
    };
    uint32_t s = blockIdx.x + gridDim.x * (uint32_t)warp;
    const uint32_t step = gridDim.x * RD.warps;
    float anc = 0.0f;
    if (s < segs) {
        const Seg g = seg_of(s, per_row, nx);
        land_codes(land, a.codes, g, width, lane);
        anc = anchor_of(g);
    }
    for (uint32_t next; s < segs; s = next) {
        const Seg g = seg_of(s, per_row, nx);
        next = next_item(s, step, segs);
        cp_async_wait_all();
        __syncwarp();
        Lane L;
#pragma unroll
        for (int i = 0; i < RUN / 8; ++i) {
            const uint4 w = reinterpret_cast<const uint4 *>(land + lane * KP)[i];
            L.cw[4 * i] = w.x;
            L.cw[4 * i + 1] = w.y;
            L.cw[4 * i + 2] = w.z;
            L.cw[4 * i + 3] = w.w;
        }
        c.closing = __shfl_sync(0xffffffffu, anc, 31);
        L.v[0] = anc;
        __syncwarp();
        if (next < segs) {
            const Seg n = seg_of(next, per_row, nx);
            land_codes(land, a.codes, n, width, lane);
            anc = anchor_of(n);
        }
        const bool full = g.x0 + SEG < nx;
        c.last = full ? SEG : nx - 1 - g.x0;
        const int in = g.valid - RUN * lane;  // in-field points of the lane
        uint32_t least = 0xffffffffu;
#pragma unroll
        for (int i = 0; i < RUN / 2; ++i) least = __vminu2(least, L.cw[i]);
        const bool zero = in > 0 && ((least & 0xffffu) == 0u || least < 0x10000u);
        if (__any_sync(0xffffffffu, zero)) {
            // outliers: their values were scattered into the output beforehand
            const float *xr = a.xrec + g.base + RUN * lane;
#pragma unroll
            for (int i = 0; i < RUN; ++i)
                if (i < in && ((i & 1) ? L.cw[i / 2] >> 16 : L.cw[i / 2] & 0xffffu) == 0u) L.v[i] = xr[i];
            levels_from<DECODE, true, false, 256>(L, c, kd.k0, kd.k1, kd.k2, 0.0f);
        } else if (full) {
            levels_from<DECODE, false, true, 256>(L, c, kd.k0, kd.k1, kd.k2, 0.0f);
        } else {
            levels_from<DECODE, false, false, 256>(L, c, kd.k0, kd.k1, kd.k2, 0.0f);
        }
        __syncwarp();  // the stage's previous contents are written out
#pragma unroll
        for (int i = 0; i < RUN / 4; ++i)
            reinterpret_cast<float4 *>(stage + lane * VP)[i] =
                make_float4(L.v[4 * i], L.v[4 * i + 1], L.v[4 * i + 2], L.v[4 * i + 3]);
        __syncwarp();
        float *dst = a.xrec + g.base;
        if (vec) {
#pragma unroll
            for (int i = 0; i < RUN / 4; ++i) {
                const int e = 4 * (32 * i + lane);
                if (e < g.valid)
                    *reinterpret_cast<float4 *>(dst + e) =
                        *reinterpret_cast<const float4 *>(stage + (e >> 5) * VP + (e & 31));
            }
        } else {
#pragma unroll 8
            for (int i = 0; i < RUN; ++i)
                if (32 * i + lane < g.valid) dst[32 * i + lane] = stage[i * VP + lane];
        }
    }
}

uint32_t segments_per_row(Dims d) { return (uint32_t)(((long long)d.nx + SEG - 1) / SEG); }

template <typename K, typename A>
cudaError_t launch_rows(K kernel, Shape shape, const A &a, size_t smem, size_t most, bool early, cudaStream_t s)
{
    // segments are fewer than 2^32 (N is), and a grid of one wave takes them in turn
    const uint32_t per_row = segments_per_row(a.dims);
    const unsigned long long segs = (unsigned long long)a.dims.nz * a.dims.ny * per_row;
    const cudaError_t e = allow_smem(kernel, most);
    if (e != cudaSuccess) return e;
    const unsigned long long wave = (unsigned long long)sm_count() * shape.ctas;
    return launch_after(early, kernel, (unsigned)(segs < wave ? segs : wave), 32 * shape.warps, smem, s, a, per_row,
                        (uint32_t)segs);
}

}  // namespace

cudaError_t launch_row_compress(const CompressArgs &a, bool early, cudaStream_t s)
{
    constexpr size_t wide = R_HIST + sizeof(uint32_t) * LANE_WINDOW;
    if (2 * a.radius > LANE_BINS) return launch_rows(k_row_compress<ENCODE_GBINS>, RC, a, wide, wide, early, s);
    return launch_rows(k_row_compress<ENCODE>, RC, a, R_HIST + sizeof(uint32_t) * 2 * (size_t)a.radius,
                       R_HIST + sizeof(uint32_t) * LANE_BINS, early, s);
}

cudaError_t launch_row_decompress(const DecompressArgs &a, bool early, cudaStream_t s)
{
    constexpr size_t smem = R_WARPS + R_WARP * RD.warps;
    return launch_rows(k_row_decompress, RD, a, smem, smem, early, s);
}

}  // namespace gi
