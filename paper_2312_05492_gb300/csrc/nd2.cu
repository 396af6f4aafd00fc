// 2-D G-Interp (Sec. IV-A: 16^2 chunks over (y, x) of every z-slice, anchors where both
// are multiples of 16, strides 8, 4, 2, 1), compression and decompression, in registers.
//
// A warp works on a strip of 64 columns (four chunks) and marches down y one chunk row
// (16 rows) at a time.  Lane (px, py) of its 8 x 4 lanes holds the 8 x 4 points at
// columns 8 px .., rows 4 py ..; so strides 1 and 2 (and 4 along x) stay inside a lane
// but for the nearest known points of its neighbours, which come by warp shuffles, and
// neither shared memory nor a barrier lies between the eight passes.  (The kernels that
// this replaced ran them over a 16 x 128 tile in shared memory, a block barrier after
// each, at 3.4 .. 4.2 warp instructions a point.)
//
// What a chunk borrows beyond its own 16 x 16 points:
//   the closing row, y = 16: the next chunk row's first row.  It depends on itself alone
//     (x passes only) and is carried to the next step, so it costs nothing: lanes py = 0
//     run the x passes on row 16 instead of row 0, which the step before left finished.
//   the closing column, x = 64, of the strip: the next strip's first column (y passes
//     only), recomputed by lanes px = 0 as a ninth column: 5 of the 40 point operations
//     a lane executes for its 32 points.
// A shuffle to the right from px = 7 wraps to px = 0, one down from py = 3 to py = 0:
// exactly the lanes that hold the closing column and the closing row.
//
// The input lands in shared memory a step ahead (cp.async), 16-byte groups permuted so
// that a warp's reads fall in distinct banks.
#include "lanes.cuh"

namespace gi {
namespace {

constexpr int PW = 8;                     // warps per CTA, each on its own strips
constexpr int P_THREADS = 32 * PW;
constexpr int P_CTAS = 2;                 // CTAs per SM: 16 warps of 128 registers (20 of 96 spill: 25% slower)
constexpr int A = 16;                     // chunk edge
constexpr int SX = 64;                    // columns of a strip
constexpr int LEVELS = 4;
// per warp: 16 landed rows and the closing column (values, or codes in the first half
// of the room), then a stage for rows that cannot be stored 16 bytes at a time
constexpr size_t P_LAND = 0;
constexpr size_t P_COL = sizeof(float) * A * SX;
constexpr size_t P_STAGE = P_COL + sizeof(float) * A;
constexpr size_t P_WARP = P_STAGE + sizeof(float) * A * SX;
constexpr size_t P_LQ = P_WARP * PW;
constexpr size_t P_SPARE = P_LQ + 16 * LEVELS;  // one word per lane for updates that count nothing
constexpr size_t P_HIST = P_SPARE + 4 * 32;
static_assert(P_WARP % 16 == 0 && P_HIST % 16 == 0, "shared layout alignment");

extern __shared__ __align__(128) unsigned char p_smem[];

enum { ROW0 = 0, ROW1 = 1, ROW2 = 2, ROW3 = 3 };

// A lane's points.  Row 0 of v is row 4 py of the chunk, but row 16 in the lanes py = 0,
// whose row 0 (finished by the previous step) is `top`.  Column 8 is the closing column
// x = 64 (lanes px = 0).  Codes: two a word; mc: the closing column's (decompression).
struct Patch {
    float v[4][9], top[9];
    uint32_t c[4][4];
    uint32_t mc[4];
};

struct Ctx : Bins {
    uint32_t cbias;
    float Rf;
    int lane, px, py;
    int lx, ly;            // last in-field column from the lane's first one, and row from the
                           // chunk's first one
    bool count0;           // row 0's codes are counted (lanes py = 0: the closing row is this run's)
    LevelQ q;
};

// Neighbour-count rule (Sec. IV-B.1).  MAYBE3: bit 0 / 1 set if x_{n-3s} / x_{n+3s} may
// lie in the chunk at all (a stencil that cannot occur is not evaluated).
template <int KIND, bool FULL, int MAYBE3>
__device__ __forceinline__ float predict(float m3, float m1, float p1, float p3, bool hm3, bool hp1, bool hp3)
{
    float p = sp_linear(m1, p1);
    if (KIND != K_LINEAR) {
        if (MAYBE3 & 2) p = hp3 ? sp_quad_right(m1, p1, p3) : p;
        if (MAYBE3 & 1) p = hm3 ? sp_quad_left(m3, m1, p1) : p;
        if ((MAYBE3 & 4)) p = hm3 && hp3 ? cubic_of<KIND>(m3, m1, p1, p3) : p;
    }
    return FULL || hp1 ? p : m1;
}

// The point in column e of row j: quantize and count (compression), or apply its code.
// active: this lane's point belongs to the pass; in: it lies in the field.
template <int MODE, bool OUTL, int J, int E>
__device__ __forceinline__ void point(Patch &P, const Ctx &c, float p, bool active, bool in)
{
    float v = P.v[J][E];
    if (MODE != DECODE) {
        const uint32_t code = quantize(v, p, c.q, c.cbias, c.Rf, v);
        if constexpr (E < 8) {
            count<MODE>(c, code, active && in && (J != ROW0 || c.count0));
            uint32_t &w = P.c[J][E / 2];
            if constexpr (E % 2 == 0) w = active ? code : w;
            else w += code << 16;  // odd columns: every lane's, after the even ones
        }
    } else {
        const uint32_t code = E == 8 ? P.mc[J] : (E % 2 ? P.c[J][(E & 7) / 2] >> 16 : P.c[J][(E & 7) / 2] & 0xffffu);
        const float xq = p + code_to_q(code, c.cbias) * c.q.twoe;
        v = OUTL && code == 0u ? v : xq;  // an outlier's stored value is there already
    }
    P.v[J][E] = active ? v : P.v[J][E];
}

__device__ __forceinline__ float from(float v, int lane) { return __shfl_sync(0xffffffffu, v, lane & 31); }

// x pass of stride S on row J.  Lanes to the right: px = 7 reads px = 0, which gives its
// closing column.
template <int MODE, bool OUTL, bool FULL, int S, int KIND, int J>
__device__ __forceinline__ void x_row(Patch &P, const Ctx &c, bool active)
{
    float *v = P.v[J];
    const int rowbase = c.lane & 24;
    const bool odd = c.px & 1;  // second half of its chunk
    const float give0 = c.px == 0 ? v[8] : v[0];
    const float next0 = from(give0, rowbase | ((c.px + 1) & 7));
    const int y = J == ROW0 ? (c.py == 0 ? A : 4 * c.py) : 4 * c.py + J;
    const bool iny = FULL || y <= c.ly;
    if constexpr (S == 8) {
        const float prev0 = from(v[0], rowbase | ((c.px - 1) & 7));
        const float p = predict<K_LINEAR, FULL, 0>(0.0f, prev0, next0, 0.0f, false, c.lx >= 8, false);
        point<MODE, OUTL, J, 0>(P, c, p, active && odd, iny && (FULL || c.lx >= 0));
    } else if constexpr (S == 4) {
        float m3 = 0.0f, p3 = 0.0f;
        if (KIND != K_LINEAR) {
            m3 = from(v[0], rowbase | ((c.px - 1) & 7));
            p3 = from(give0, rowbase | ((c.px + 2) & 7));
        }
        const float p = predict<KIND, FULL, 3>(m3, v[0], next0, p3, odd, c.lx >= 8, !odd && (FULL || c.lx >= 16));
        point<MODE, OUTL, J, 4>(P, c, p, active, iny && (FULL || c.lx >= 4));
    } else if constexpr (S == 2) {
        float m3 = 0.0f, p3 = 0.0f;
        if (KIND != K_LINEAR) {
            m3 = from(v[4], rowbase | ((c.px - 1) & 7));
            p3 = from(v[4], rowbase | ((c.px + 1) & 7));
        }
        const float k0 = v[0], k4 = v[4];
        point<MODE, OUTL, J, 2>(P, c, predict<KIND, FULL, 7>(m3, k0, k4, next0, odd, c.lx >= 4, FULL || c.lx >= 8),
                                    active, iny && (FULL || c.lx >= 2));
        point<MODE, OUTL, J, 6>(
            P, c, predict<KIND, FULL, 7>(k0, k4, next0, p3, true, c.lx >= 8, !odd && (FULL || c.lx >= 12)), active,
            iny && (FULL || c.lx >= 6));
    } else {
        float m3 = 0.0f, p3 = 0.0f;
        if (KIND != K_LINEAR) {
            m3 = from(v[6], rowbase | ((c.px - 1) & 7));
            p3 = from(v[2], rowbase | ((c.px + 1) & 7));
        }
        const float k0 = v[0], k2 = v[2], k4 = v[4], k6 = v[6];
        point<MODE, OUTL, J, 1>(P, c, predict<KIND, FULL, 7>(m3, k0, k2, k4, odd, c.lx >= 2, FULL || c.lx >= 4),
                                    active, iny && (FULL || c.lx >= 1));
        point<MODE, OUTL, J, 3>(P, c, predict<KIND, FULL, FULL ? 4 : 7>(k0, k2, k4, k6, true, c.lx >= 4, FULL || c.lx >= 6),
                                    active, iny && (FULL || c.lx >= 3));
        point<MODE, OUTL, J, 5>(P, c, predict<KIND, FULL, FULL ? 4 : 7>(k2, k4, k6, next0, true, c.lx >= 6, FULL || c.lx >= 8),
                                    active, iny && (FULL || c.lx >= 5));
        point<MODE, OUTL, J, 7>(
            P, c, predict<KIND, FULL, 7>(k4, k6, next0, p3, true, c.lx >= 8, !odd && (FULL || c.lx >= 10)), active,
            iny && (FULL || c.lx >= 7));
    }
}

// The x pass of stride S on the rows that are multiples of M.
template <int MODE, bool OUTL, bool FULL, int S, int KIND, int M>
__device__ __forceinline__ void x_pass(Patch &P, const Ctx &c)
{
    const bool row0 = M == 16 ? c.py == 0 : (M == 8 ? (c.py & 1) == 0 : true);
    x_row<MODE, OUTL, FULL, S, KIND, ROW0>(P, c, row0);
    if constexpr (M <= 2) x_row<MODE, OUTL, FULL, S, KIND, ROW2>(P, c, true);
    if constexpr (M == 1) {
        x_row<MODE, OUTL, FULL, S, KIND, ROW1>(P, c, true);
        x_row<MODE, OUTL, FULL, S, KIND, ROW3>(P, c, true);
    }
}

// y pass of stride S in column E.  Lanes below: py = 3 reads py = 0, whose row 0 is the
// closing row.
template <int MODE, bool OUTL, bool FULL, int S, int KIND, int E>
__device__ __forceinline__ void y_col(Patch &P, const Ctx &c, bool active)
{
    const bool inx = FULL || E <= c.lx;
    const float x0 = P.v[ROW0][E];
    const float own0 = c.py == 0 ? P.top[E] : x0;  // row 4 py
    if constexpr (S == 8) {
        const float m1 = from(own0, c.lane - 16), p1 = from(x0, c.lane + 16);
        const float p = predict<K_LINEAR, FULL, 0>(0.0f, m1, p1, 0.0f, false, c.ly >= 16, false);
        point<MODE, OUTL, ROW0, E>(P, c, p, active && c.py == 2, inx && (FULL || c.ly >= 8));
    } else if constexpr (S == 4) {
        const float m1 = from(own0, c.lane - 8), p1 = from(x0, c.lane + 8);
        float m3 = 0.0f, p3 = 0.0f;
        if (KIND != K_LINEAR) {
            m3 = from(own0, c.lane - 24);
            p3 = from(x0, c.lane + 24);
        }
        const float p = predict<KIND, FULL, 3>(m3, m1, p1, p3, c.py == 3, 4 * c.py + 4 <= c.ly,
                                               c.py == 1 && (FULL || c.ly >= 16));
        point<MODE, OUTL, ROW0, E>(P, c, p, active && (c.py & 1), inx && (FULL || 4 * c.py <= c.ly));
    } else {
        const float below0 = from(x0, c.lane + 8);  // row 4 py + 4
        if constexpr (S == 2) {
            float m3 = 0.0f, p3 = 0.0f;
            if (KIND != K_LINEAR) {
                m3 = from(own0, c.lane - 8);
                p3 = from(x0, c.lane + 16);
            }
            const int y = 4 * c.py + 2;
            const float p = predict<KIND, FULL, 7>(m3, own0, below0, p3, c.py > 0, y + 2 <= c.ly,
                                                   c.py < 3 && (FULL || y + 6 <= c.ly));
            point<MODE, OUTL, ROW2, E>(P, c, p, active, inx && (FULL || y <= c.ly));
        } else {
            const float r2 = P.v[ROW2][E];
            float m3 = 0.0f, p3 = 0.0f;
            if (KIND != K_LINEAR) {
                m3 = from(r2, c.lane - 8);
                p3 = from(r2, c.lane + 8);
            }
            const int y = 4 * c.py;
            point<MODE, OUTL, ROW1, E>(P, c, predict<KIND, FULL, 7>(m3, own0, r2, below0, c.py > 0, y + 2 <= c.ly,
                                                                     FULL || y + 4 <= c.ly),
                                           active, inx && (FULL || y + 1 <= c.ly));
            point<MODE, OUTL, ROW3, E>(P, c, predict<KIND, FULL, 7>(own0, r2, below0, p3, true, y + 4 <= c.ly,
                                                                     c.py < 3 && (FULL || y + 6 <= c.ly)),
                                           active, inx && (FULL || y + 3 <= c.ly));
        }
    }
}

// The y pass of stride S in the columns that are multiples of M, and the closing column.
template <int MODE, bool OUTL, bool FULL, int S, int KIND, int M>
__device__ __forceinline__ void y_pass(Patch &P, const Ctx &c)
{
    y_col<MODE, OUTL, FULL, S, KIND, 0>(P, c, M == 16 ? (c.px & 1) == 0 : true);
    if constexpr (M <= 4) y_col<MODE, OUTL, FULL, S, KIND, 4>(P, c, true);
    if constexpr (M <= 2) {
        y_col<MODE, OUTL, FULL, S, KIND, 2>(P, c, true);
        y_col<MODE, OUTL, FULL, S, KIND, 6>(P, c, true);
    }
    if constexpr (M == 1) {
        y_col<MODE, OUTL, FULL, S, KIND, 1>(P, c, true);
        y_col<MODE, OUTL, FULL, S, KIND, 3>(P, c, true);
        y_col<MODE, OUTL, FULL, S, KIND, 5>(P, c, true);
        y_col<MODE, OUTL, FULL, S, KIND, 7>(P, c, true);
    }
    y_col<MODE, OUTL, FULL, S, KIND, 8>(P, c, true);
}

// Kinds of the level classes (strides 1, 2, 4 and 8) along y and x.
struct Kinds {
    int y[3], x[3];
};
__device__ __forceinline__ Kinds kinds_of(const interp_header *h)
{
    Kinds k;
    const int ky = h->cfg.cubic_kind[1] ? K_NATURAL : K_NAK, kx = h->cfg.cubic_kind[2] ? K_NATURAL : K_NAK;
#pragma unroll
    for (int l = 0; l < 3; ++l) {
        k.y[l] = h->cfg.level_kind[l] ? ky : K_LINEAR;
        k.x[l] = h->cfg.level_kind[l] ? kx : K_LINEAR;
    }
    return k;
}

template <int MODE, bool OUTL, bool FULL, int S, bool XFIRST>
__device__ __forceinline__ void x_any(Patch &P, const Ctx &c, int kind)
{
    constexpr int M = XFIRST ? 2 * S : S;
    // inside a chunk stride 8 is always linear, and stride 4 has no cubic stencil
    if (S == 8 || kind == K_LINEAR) x_pass<MODE, OUTL, FULL, S, K_LINEAR, M>(P, c);
    else if (S == 4 || kind == K_NAK) x_pass<MODE, OUTL, FULL, S, K_NAK, M>(P, c);
    else x_pass<MODE, OUTL, FULL, S, S <= 2 ? K_NATURAL : K_LINEAR, M>(P, c);
}
template <int MODE, bool OUTL, bool FULL, int S, bool XFIRST>
__device__ __forceinline__ void y_any(Patch &P, const Ctx &c, int kind)
{
    constexpr int M = XFIRST ? S : 2 * S;
    if (S == 8 || kind == K_LINEAR) y_pass<MODE, OUTL, FULL, S, K_LINEAR, M>(P, c);
    else if (S == 4 || kind == K_NAK) y_pass<MODE, OUTL, FULL, S, K_NAK, M>(P, c);
    else y_pass<MODE, OUTL, FULL, S, S <= 2 ? K_NATURAL : K_LINEAR, M>(P, c);
}

template <int MODE, bool OUTL, bool FULL, int S, bool XFIRST>
__device__ __forceinline__ void levels_from(Patch &P, Ctx &c, const Kinds &k)
{
    constexpr int l = S == 8 ? 3 : (S == 4 ? 2 : (S == 2 ? 1 : 0));
    const float4 q = reinterpret_cast<const float4 *>(p_smem + P_LQ)[l];
    c.q = LevelQ{q.x, q.y, q.z};
    const int kx = k.x[l < 2 ? l : 2], ky = k.y[l < 2 ? l : 2];  // stride 8 follows stride 4
    if (XFIRST) {
        x_any<MODE, OUTL, FULL, S, true>(P, c, kx);
        y_any<MODE, OUTL, FULL, S, true>(P, c, ky);
    } else {
        y_any<MODE, OUTL, FULL, S, false>(P, c, ky);
        x_any<MODE, OUTL, FULL, S, false>(P, c, kx);
    }
    if constexpr (S > 1) levels_from<MODE, OUTL, FULL, S / 2, XFIRST>(P, c, k);
}

// A run's first row on its own (it has no step before it): the x passes on row 0 of the
// lanes py = 0, as the closing row of a chunk row above.
template <int MODE, int S>
__device__ __forceinline__ void first_row_from(Patch &P, Ctx &c, const Kinds &k)
{
    constexpr int l = S == 8 ? 3 : (S == 4 ? 2 : (S == 2 ? 1 : 0));
    const float4 q = reinterpret_cast<const float4 *>(p_smem + P_LQ)[l];
    c.q = LevelQ{q.x, q.y, q.z};
    const int kx = k.x[l < 2 ? l : 2];
    if (S == 8 || kx == K_LINEAR) x_pass<MODE, true, false, S, K_LINEAR, 16>(P, c);
    else if (S == 4 || kx == K_NAK) x_pass<MODE, true, false, S, K_NAK, 16>(P, c);
    else x_pass<MODE, true, false, S, S <= 2 ? K_NATURAL : K_LINEAR, 16>(P, c);
    if constexpr (S > 1) first_row_from<MODE, S / 2>(P, c, k);
}

// ------------------------------------------------------------ work items
// Items: (run of chunk rows, slice) x strip, strips fastest.
struct Plan {
    uint32_t strips, runs, items;  // per slice: strips, runs; items in all
    int run, rows;                 // chunk rows per run, chunk rows per slice
};
struct Item {
    int z, x0, r0, r1;  // slice, first column, chunk rows [r0, r1)
};
__device__ __forceinline__ Item item_of(const Plan &p, uint32_t i)
{
    Item t;
    const uint32_t a = i / p.strips, z = a / p.runs;
    t.x0 = (int)(i - a * p.strips) * SX;
    t.z = (int)z;
    t.r0 = (int)(a - z * p.runs) * p.run;
    t.r1 = min(t.r0 + p.run, p.rows);
    return t;
}

// 16-byte group g (of 16) of a landed row of values: even groups first, so that the 8
// lanes px of a row read 128 consecutive bytes twice
__device__ __forceinline__ int slot_of(int g) { return (g >> 1) + 8 * (g & 1); }

// ------------------------------------------------------------ compression
// Rows y0 + 1 .. y0 + 16 of a strip, columns x0 .. x0 + 64.
__device__ __forceinline__ void land_values(unsigned char *land, const float *x, Dims d, int z, int y0, int x0, bool vec,
                                            int lane)
{
    float *dst = reinterpret_cast<float *>(land + P_LAND);
    const float *src = x + ((size_t)z * d.ny + y0 + 1) * d.nx + x0;
    const int ny = d.ny - 1 - y0, nx = d.nx - x0;  // rows, columns there are
    if (vec) {
        const int g = lane & 15;
#pragma unroll
        for (int i = 0; i < A / 2; ++i) {
            const int r = 2 * i + (lane >> 4);
            if (r < ny && 4 * g < nx) cp_async16(dst + r * SX + 4 * slot_of(g), src + (size_t)r * d.nx + 4 * g);
        }
    } else {
#pragma unroll 4
        for (int i = 0; i < 2 * A; ++i) {
            const int r = i >> 1, e = 32 * (i & 1) + lane;
            if (r < ny && e < nx) cp_async4(dst + r * SX + 4 * slot_of(e >> 2) + (e & 3), src + (size_t)r * d.nx + e);
        }
    }
    if (lane < A && lane < ny && SX < nx)
        cp_async4(reinterpret_cast<float *>(land + P_COL) + lane, src + (size_t)lane * d.nx + SX);
    cp_async_commit();
}

__device__ __forceinline__ void read_row(float (&v)[9], const unsigned char *land, int r, int px)
{
    const float4 *row = reinterpret_cast<const float4 *>(land + P_LAND) + r * (SX / 4);
    const float4 a = row[px], b = row[px + 8];
    v[0] = a.x;
    v[1] = a.y;
    v[2] = a.z;
    v[3] = a.w;
    v[4] = b.x;
    v[5] = b.y;
    v[6] = b.z;
    v[7] = b.w;
    v[8] = reinterpret_cast<const float *>(land + P_COL)[r];
}

__device__ __forceinline__ void set_rows_codes(Patch &P, uint32_t R)
{
#pragma unroll
    for (int j = 0; j < 4; ++j) P.c[j][0] = R;  // column 0 of even px in row 0: an anchor, code R
}

template <int MODE>
__global__ void __launch_bounds__(P_THREADS, P_CTAS) k_plane_compress(const CompressArgs a, const Plan plan)
{
    wait_for_previous();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Dims d = a.dims;
    const int bins = MODE == ENCODE_GBINS ? LANE_WINDOW : 2 * a.radius;  // in shared memory
    const int win0 = MODE == ENCODE_GBINS ? a.radius - LANE_WINDOW / 2 : 0;
    uint32_t *hs = reinterpret_cast<uint32_t *>(p_smem + P_HIST);
    store_levels<LEVELS>(a.hdr, reinterpret_cast<float4 *>(p_smem + P_LQ));
    for (int i = threadIdx.x; i < bins; i += P_THREADS) hs[i] = 0u;
    __syncthreads();
    unsigned char *land = p_smem + P_WARP * warp;
    uint16_t *stage = reinterpret_cast<uint16_t *>(land + P_STAGE);
    const bool vec = (d.nx & 3) == 0 && (reinterpret_cast<uintptr_t>(a.x) & 15u) == 0;
    const bool vec_codes = (d.nx & 7) == 0 && (reinterpret_cast<uintptr_t>(a.codes) & 15u) == 0;
    const Kinds kd = kinds_of(a.hdr);
    const interp_header *h = a.hdr;
    const int o0 = h->cfg.dim_order[0], o1 = h->cfg.dim_order[1];
    const bool xfirst = o0 == 2 || (o1 == 2 && o0 == 0);  // x before y
    const int wpr = (d.nx + 31) / 32, ax = (d.nx - 1) / A + 1, ay = (d.ny - 1) / A + 1;
    Ctx c;
    c.cbias = kMagicBits - (uint32_t)a.radius;
    c.R = (uint32_t)a.radius;
    c.Rf = (float)a.radius;
    c.hist = smem_u32(hs);
    c.win0 = (uint32_t)win0;
    c.spare = smem_u32(p_smem + P_SPARE) + 4u * lane;
    c.hist_g = a.hist;
    c.lane = lane;
    c.px = lane & 7;
    c.py = lane >> 3;

    const uint32_t step = gridDim.x * PW;
    // items go to CTAs first, then to their warps: few items spread over the SMs
    for (uint32_t it = blockIdx.x + gridDim.x * (uint32_t)warp; it < plan.items; it += step) {
        const Item t = item_of(plan, it);
        __syncwarp();
        land_values(land, a.x, d, t.z, A * t.r0, t.x0, vec, lane);
        c.lx = d.nx - 1 - t.x0 - 8 * c.px;
        Patch P;
        uint32_t tc[4];  // codes of row 0 (lanes py = 0)
        {                // the run's first row
            const int y0 = A * t.r0;
            const float *src = a.x + ((size_t)t.z * d.ny + y0) * d.nx + t.x0 + 8 * c.px;
#pragma unroll
            for (int e = 0; e < 8; ++e) P.v[ROW0][e] = c.py == 0 && e <= c.lx ? __ldg(src + e) : 0.0f;
            P.v[ROW0][8] = lane == 0 && t.x0 + SX < d.nx ? __ldg(src + SX) : 0.0f;
            P.c[ROW0][0] = c.R;
            c.ly = A;  // the row as row 16 of a chunk row that has it
            c.count0 = c.py == 0;
            first_row_from<MODE, 8>(P, c, kd);
        }
        for (int r = t.r0; r < t.r1; ++r) {
            const int y0 = A * r;
            // the closing row becomes the first row
#pragma unroll
            for (int e = 0; e < 9; ++e) P.top[e] = P.v[ROW0][e];
#pragma unroll
            for (int w = 0; w < 4; ++w) tc[w] = P.c[ROW0][w];
            cp_async_wait_all();
            __syncwarp();
            read_row(P.v[ROW0], land, c.py == 0 ? A - 1 : 4 * c.py - 1, c.px);
            read_row(P.v[ROW1], land, 4 * c.py, c.px);
            read_row(P.v[ROW2], land, 4 * c.py + 1, c.px);
            read_row(P.v[ROW3], land, 4 * c.py + 2, c.px);
            __syncwarp();
            if (r + 1 < t.r1) land_values(land, a.x, d, t.z, y0 + A, t.x0, vec, lane);  // lands during the passes
            set_rows_codes(P, c.R);
            c.ly = d.ny - 1 - y0;
            c.count0 = c.py != 0 || r + 1 < t.r1;
            const bool full = d.nx - 1 - t.x0 >= SX && c.ly >= A;
            if (full) {
                if (xfirst) levels_from<MODE, false, true, 8, true>(P, c, kd);
                else levels_from<MODE, false, true, 8, false>(P, c, kd);
            } else {
                if (xfirst) levels_from<MODE, false, false, 8, true>(P, c, kd);
                else levels_from<MODE, false, false, 8, false>(P, c, kd);
            }
            // owned rows: row 0 of the lanes py = 0 is the one carried in
            uint32_t out[4][4];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                out[0][w] = c.py == 0 ? tc[w] : P.c[0][w];
#pragma unroll
                for (int j = 1; j < 4; ++j) out[j][w] = P.c[j][w];
            }
            if (c.py == 0 && (c.px & 1) == 0 && c.lx >= 0)
                a.anchors[((size_t)t.z * ay + r) * ax + (t.x0 + 8 * c.px) / A] = P.top[0];
            uint32_t least = 0xffffffffu;
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int w = 0; w < 4; ++w) least = __vminu2(least, out[j][w]);
            const bool any = __any_sync(0xffffffffu, (least & 0xffffu) == 0u || least < 0x10000u);
            const int rows = min(4, c.ly + 1 - 4 * c.py);  // in-field rows of the lane (may be negative)
            const size_t grow = (size_t)t.z * d.ny + y0 + 4 * c.py;
            // outlier words (row-major bitmap): a row's 64 columns are two words, 4 lanes each
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t word = 0u;
                if (any) {
                    uint32_t z8 = 0u;
#pragma unroll
                    for (int w = 0; w < 4; ++w)
                        z8 |= ((out[j][w] & 0xffffu) == 0u ? 1u : 0u) << (2 * w) |
                              (out[j][w] < 0x10000u ? 2u : 0u) << (2 * w);
                    if (c.lx < 7) z8 &= c.lx >= 0 ? (2u << c.lx) - 1u : 0u;
                    word = z8 << (8 * (c.px & 3));
                    word |= __shfl_xor_sync(0xffffffffu, word, 1);
                    word |= __shfl_xor_sync(0xffffffffu, word, 2);
                }
                if ((c.px & 3) == 0 && j < rows && c.lx >= 0) {
                    const size_t gw = (grow + j) * wpr + (t.x0 + 8 * c.px) / 32;
                    a.bitmap[gw] = word;
                    if (word) atomicAdd(a.blockcnt + gw / BITMAP_BLOCK_WORDS, (uint32_t)__popc(word));
                }
            }
            if (vec_codes) {
                if (c.lx >= 0)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (j < rows)
                            *reinterpret_cast<uint4 *>(a.codes + (grow + j) * d.nx + t.x0 + 8 * c.px) =
                                make_uint4(out[j][0], out[j][1], out[j][2], out[j][3]);
            } else {  // rows that are not 16-byte aligned: through shared memory, one code per lane
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    *reinterpret_cast<uint4 *>(stage + (4 * c.py + j) * SX + 8 * c.px) =
                        make_uint4(out[j][0], out[j][1], out[j][2], out[j][3]);
                __syncwarp();
                uint16_t *dst = a.codes + ((size_t)t.z * d.ny + y0) * d.nx + t.x0;
                const int ny = min(A, d.ny - y0), nx = d.nx - t.x0;
#pragma unroll 4
                for (int i = 0; i < 2 * ny; ++i) {
                    const int y = i >> 1, e = 32 * (i & 1) + lane;
                    if (e < nx) dst[(size_t)y * d.nx + e] = stage[y * SX + e];
                }
            }
        }
    }
    if (a.hist) {
        __syncthreads();
        for (int i = threadIdx.x; i < bins; i += P_THREADS)
            if (hs[i]) atomicAdd(&a.hist[win0 + i], hs[i]);
    }
}

// ---------------------------------------------------------- decompression
// Codes of rows y0 + 1 .. y0 + 16, columns x0 .. x0 + 64.
// Returns the closing column's code of row y0 + 1 + lane (lanes 0 .. 15), a load that is
// first needed when the landed rows are.
__device__ __forceinline__ uint32_t land_codes(unsigned char *land, const uint16_t *codes, Dims d, int z, int y0,
                                               int x0, int width, int lane)
{
    uint16_t *dst = reinterpret_cast<uint16_t *>(land + P_LAND);
    const uint16_t *src = codes + ((size_t)z * d.ny + y0 + 1) * d.nx + x0;
    const int ny = d.ny - 1 - y0, nx = d.nx - x0;
    if (width == 8) {
#pragma unroll
        for (int i = 0; i < A / 4; ++i) {
            const int r = 4 * i + (lane >> 3), e = 8 * (lane & 7);
            if (r < ny && e < nx) cp_async16(dst + r * SX + e, src + (size_t)r * d.nx + e);
        }
    } else if (width == 2) {
#pragma unroll 4
        for (int r = 0; r < A; ++r)
            if (r < ny && 2 * lane < nx) cp_async4(dst + r * SX + 2 * lane, src + (size_t)r * d.nx + 2 * lane);
    } else {
#pragma unroll 4
        for (int i = 0; i < 2 * A; ++i) {
            const int r = i >> 1, e = 32 * (i & 1) + lane;
            if (r < ny && e < nx) dst[r * SX + e] = __ldg(src + (size_t)r * d.nx + e);
        }
    }
    cp_async_commit();
    return lane < A && lane < ny && SX < nx ? __ldg(src + (size_t)lane * d.nx + SX) : 0u;
}

__global__ void __launch_bounds__(P_THREADS, P_CTAS) k_plane_decompress(const DecompressArgs a, const Plan plan)
{
    wait_for_previous();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Dims d = a.dims;
    store_levels<LEVELS>(a.hdr, reinterpret_cast<float4 *>(p_smem + P_LQ));
    __syncthreads();
    unsigned char *land = p_smem + P_WARP * warp;
    float *stage = reinterpret_cast<float *>(land + P_STAGE);
    const uintptr_t ca = reinterpret_cast<uintptr_t>(a.codes);
    const int width = (d.nx & 7) == 0 && (ca & 15u) == 0 ? 8 : ((d.nx & 1) == 0 && (ca & 3u) == 0 ? 2 : 1);
    const uintptr_t xa = reinterpret_cast<uintptr_t>(a.xrec);
    const int vec = (d.nx & 7) == 0 && (xa & 31u) == 0 ? 8 : ((d.nx & 3) == 0 && (xa & 15u) == 0 ? 4 : 1);
    const interp_header *h = a.hdr;
    const Kinds kd = kinds_of(h);
    const int o0 = h->cfg.dim_order[0], o1 = h->cfg.dim_order[1];
    const bool xfirst = o0 == 2 || (o1 == 2 && o0 == 0);
    const int ax = (d.nx - 1) / A + 1, ay = (d.ny - 1) / A + 1;
    Ctx c;
    c.R = (uint32_t)h->cfg.radius;
    c.cbias = kMagicBits - c.R;
    c.Rf = 0.0f;
    c.hist = c.spare = c.win0 = 0u;
    c.hist_g = nullptr;
    c.count0 = false;
    c.lane = lane;
    c.px = lane & 7;
    c.py = lane >> 3;

    // anchors of chunk row r: columns 8 px of the strip (even px), and x = 64 (in v8, lane 0)
    auto anchors_of = [&](int z, int r, int x0, float &v0, float &v8) {
        const float *row = a.anchors + ((size_t)z * ay + r) * ax + x0 / A;
        v0 = v8 = 0.0f;
        if (r < ay && c.py == 0 && (c.px & 1) == 0 && x0 + 8 * c.px < d.nx) v0 = __ldg(row + c.px / 2);
        if (r < ay && lane == 0 && x0 + SX < d.nx) v8 = __ldg(row + SX / A);
    };
    // outliers of a row: their values were scattered into the output beforehand
    auto outliers_of = [&](Patch &P, int j, const float *row, bool in) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const uint32_t code = e & 1 ? P.c[j][e / 2] >> 16 : P.c[j][e / 2] & 0xffffu;
            if (in && code == 0u && e <= c.lx) P.v[j][e] = row[e];
        }
    };

    const uint32_t step = gridDim.x * PW;
    for (uint32_t it = blockIdx.x + gridDim.x * (uint32_t)warp; it < plan.items; it += step) {
        const Item t = item_of(plan, it);
        __syncwarp();
        uint32_t col = land_codes(land, a.codes, d, t.z, A * t.r0, t.x0, width, lane);
        c.lx = d.nx - 1 - t.x0 - 8 * c.px;
        Patch P;
        {  // the run's first row
            const size_t g = ((size_t)t.z * d.ny + A * t.r0) * d.nx + t.x0 + 8 * c.px;
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const bool in = c.py == 0;
                const uint32_t lo = in && 2 * w <= c.lx ? __ldg(a.codes + g + 2 * w) : c.R;
                const uint32_t hi = in && 2 * w + 1 <= c.lx ? __ldg(a.codes + g + 2 * w + 1) : c.R;
                P.c[ROW0][w] = lo | (hi << 16);
            }
            P.mc[ROW0] = c.R;
            anchors_of(t.z, t.r0, t.x0, P.v[ROW0][0], P.v[ROW0][8]);
#pragma unroll
            for (int e = 1; e < 8; ++e) P.v[ROW0][e] = 0.0f;
            outliers_of(P, ROW0, a.xrec + g, c.py == 0);
            c.ly = A;
            first_row_from<DECODE, 8>(P, c, kd);
        }
        float anc0, anc8;
        anchors_of(t.z, t.r0 + 1, t.x0, anc0, anc8);
        for (int r = t.r0; r < t.r1; ++r) {
            const int y0 = A * r;
#pragma unroll
            for (int e = 0; e < 9; ++e) P.top[e] = P.v[ROW0][e];
            cp_async_wait_all();
            __syncwarp();
            const int r0 = c.py == 0 ? A - 1 : 4 * c.py - 1;  // landed row of this lane's row 0
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int lr = j == 0 ? r0 : 4 * c.py + j - 1;
                const uint4 w = *reinterpret_cast<const uint4 *>(land + P_LAND + 2 * (lr * SX + 8 * c.px));
                P.c[j][0] = w.x;
                P.c[j][1] = w.y;
                P.c[j][2] = w.z;
                P.c[j][3] = w.w;
                P.mc[j] = __shfl_sync(0xffffffffu, col, lr);
            }
            P.v[ROW0][0] = anc0;  // anchors of the closing row (lanes py = 0)
            P.v[ROW0][8] = anc8;
            __syncwarp();
            if (r + 1 < t.r1) {
                col = land_codes(land, a.codes, d, t.z, y0 + A, t.x0, width, lane);
                anchors_of(t.z, r + 2, t.x0, anc0, anc8);
            }
            c.ly = d.ny - 1 - y0;
            const bool colin = c.px == 0 && t.x0 + SX < d.nx;  // the closing column is this lane's and in the field
            const int rows = min(4, c.ly + 1 - 4 * c.py);      // in-field rows of the lane (may be negative)
            const bool in0 = c.py == 0 ? c.ly >= A : rows > 0;
            uint32_t least = 0xffffffffu;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (!(j == 0 ? in0 : j < rows)) continue;
#pragma unroll
                for (int w = 0; w < 4; ++w) least = __vminu2(least, P.c[j][w]);
                if (colin) least = __vminu2(least, P.mc[j] | 0xffff0000u);
            }
            if (c.lx < 0 && !colin) least = 0xffffffffu;
            const bool full = d.nx - 1 - t.x0 >= SX && c.ly >= A;
            if (__any_sync(0xffffffffu, (least & 0xffffu) == 0u || least < 0x10000u)) {
                const float *base = a.xrec + ((size_t)t.z * d.ny + y0) * d.nx + t.x0;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool in = j == 0 ? in0 : j < rows;
                    const int y = j == 0 && c.py == 0 ? A : 4 * c.py + j;
                    outliers_of(P, j, base + (size_t)y * d.nx + 8 * c.px, in);
                    if (in && colin && P.mc[j] == 0u) P.v[j][8] = base[(size_t)y * d.nx + SX];
                }
                if (xfirst) levels_from<DECODE, true, false, 8, true>(P, c, kd);
                else levels_from<DECODE, true, false, 8, false>(P, c, kd);
            } else if (full) {
                if (xfirst) levels_from<DECODE, false, true, 8, true>(P, c, kd);
                else levels_from<DECODE, false, true, 8, false>(P, c, kd);
            } else {
                if (xfirst) levels_from<DECODE, false, false, 8, true>(P, c, kd);
                else levels_from<DECODE, false, false, 8, false>(P, c, kd);
            }
            float *dst = a.xrec + ((size_t)t.z * d.ny + y0) * d.nx + t.x0;
            float o[8];
            if (vec != 1) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) o[e] = j == 0 && c.py == 0 ? P.top[e] : P.v[j][e];
                    if (j >= rows) continue;
                    float *g = dst + (size_t)(4 * c.py + j) * d.nx + 8 * c.px;
                    if (vec == 8) {
                        if (c.lx >= 0)  // 32 bytes a lane: whole sectors
                            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(g),
                                         "f"(o[0]), "f"(o[1]), "f"(o[2]), "f"(o[3]), "f"(o[4]), "f"(o[5]), "f"(o[6]),
                                         "f"(o[7])
                                         : "memory");
                    } else {
                        if (c.lx >= 0) reinterpret_cast<float4 *>(g)[0] = make_float4(o[0], o[1], o[2], o[3]);
                        if (c.lx >= 4) reinterpret_cast<float4 *>(g)[1] = make_float4(o[4], o[5], o[6], o[7]);
                    }
                }
            } else {  // unaligned rows: through shared memory, one value per lane
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) o[e] = j == 0 && c.py == 0 ? P.top[e] : P.v[j][e];
                    float4 *row = reinterpret_cast<float4 *>(stage) + (4 * c.py + j) * (SX / 4);
                    row[c.px] = make_float4(o[0], o[1], o[2], o[3]);
                    row[c.px + 8] = make_float4(o[4], o[5], o[6], o[7]);
                }
                __syncwarp();
                const int ny = min(A, d.ny - y0), nx = d.nx - t.x0;
#pragma unroll 4
                for (int i = 0; i < 2 * ny; ++i) {
                    const int y = i >> 1, e = 32 * (i & 1) + lane;
                    if (e < nx) dst[(size_t)y * d.nx + e] = stage[y * SX + 4 * slot_of(e >> 2) + (e & 3)];
                }
            }
        }
    }
}

// Chunk rows per run: the busiest warp's steps, each run costing a third of a step for
// its first row, must be few; ties to the longer run.
Plan plan_of(Dims d, unsigned long long warps)
{
    Plan p;
    p.rows = (d.ny + A - 1) / A;
    p.strips = (uint32_t)((d.nx + SX - 1) / SX);
    double best = 1e300;
    p.run = p.rows;
    for (int run = 1; run <= p.rows; run = run < 8 ? run + 1 : run + run / 8) {
        const unsigned long long items = (unsigned long long)d.nz * p.strips * ((p.rows + run - 1) / run);
        const double cost = (double)((items + warps - 1) / warps) * (run + 0.35);
        if (cost <= best) {
            best = cost;
            p.run = run;
        }
    }
    p.runs = (uint32_t)((p.rows + p.run - 1) / p.run);
    p.items = (uint32_t)((unsigned long long)d.nz * p.strips * p.runs);
    return p;
}

template <typename K, typename Args>
cudaError_t launch_planes(K kernel, const Args &a, size_t smem, size_t most, bool early, cudaStream_t s)
{
    const cudaError_t e = allow_smem(kernel, most);
    if (e != cudaSuccess) return e;
    const uint32_t wave = (uint32_t)(sm_count() * P_CTAS);
    const Plan p = plan_of(a.dims, (unsigned long long)wave * PW);
    return launch_after(early, kernel, p.items < wave ? p.items : wave, P_THREADS, smem, s, a, p);
}

}  // namespace

cudaError_t launch_plane_compress(const CompressArgs &a, bool early, cudaStream_t s)
{
    constexpr size_t wide = P_HIST + sizeof(uint32_t) * LANE_WINDOW;
    if (2 * a.radius > LANE_BINS) return launch_planes(k_plane_compress<ENCODE_GBINS>, a, wide, wide, early, s);
    return launch_planes(k_plane_compress<ENCODE>, a, P_HIST + sizeof(uint32_t) * 2 * (size_t)a.radius,
                         P_HIST + sizeof(uint32_t) * LANE_BINS, early, s);
}

cudaError_t launch_plane_decompress(const DecompressArgs &a, bool early, cudaStream_t s)
{
    return launch_planes(k_plane_decompress, a, P_HIST, P_HIST, early, s);
}

}  // namespace gi
