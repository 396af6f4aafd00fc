// What the 1-D and the 2-D kernels share: their modes and stencil kinds, the level constants,
// and the histogram.
#pragma once
#include "tma.cuh"

namespace gi {
namespace {

// What a kernel does with the points: apply the stored codes; quantize and count in shared
// memory, or (more than LANE_BINS bins) partly in global memory.
enum { DECODE = 0, ENCODE = 1, ENCODE_GBINS = 2 };
enum { K_LINEAR = 0, K_NAK = 1, K_NATURAL = 2 };
constexpr int LANE_BINS = 8192;    // bins kept in shared memory
constexpr int LANE_WINDOW = 2048;  // and with more than those, the bins around R

// Level constants, one thread per level, with the header's own arithmetic (alpha^l by
// repeated multiplication in double).
template <int LEVELS>
__device__ __forceinline__ void store_levels(const interp_header *h, float4 *lq)
{
    const int l = threadIdx.x;
    if (l >= LEVELS) return;
    double apow = 1.0;
    for (int j = 0; j < l; ++j) apow *= h->alpha;
    const float e = (float)(h->eb_abs / apow);
    lq[l] = make_float4(e, 2.0f * e, (float)(1.0 / (2.0 * (double)e)), 0.0f);
}

template <int KIND>
__device__ __forceinline__ float cubic_of(float m3, float m1, float p1, float p3)
{
    return KIND == K_NATURAL ? sp_cubic_nat_call(m3, m1, p1, p3) : sp_cubic_nak(m3, m1, p1, p3);
}

// Where codes are counted.
struct Bins {
    uint32_t R;
    uint32_t hist, spare;  // shared addresses of the bins (of bin win0's) and of this lane's spare word
    uint32_t win0;         // first bin kept in shared memory
    uint32_t *hist_g;      // all bins in global memory, may be null
};

// Count a code other than R (whose bin is filled in afterwards as N minus the others).
// ENCODE_GBINS: more bins than shared memory keeps.  Those around R are kept there all the
// same (nearly all codes, and few bins: in global memory their updates wait for one another;
// 64 x 2^17 points, radius 4097, bound 1e-5: 893 -> 25 us; 8 x 2048 x 2048 points, bound
// 1e-3: 4.49 -> 0.13 ms); the others are counted in global memory.
template <int MODE>
__device__ __forceinline__ void count(const Bins &c, uint32_t code, bool counts)
{
    const bool yes = counts && code != c.R;
    if constexpr (MODE == ENCODE_GBINS) {
        const uint32_t w = code - c.win0;
        const bool in = w < (uint32_t)LANE_WINDOW;
        asm volatile("red.shared.add.u32 [%0], 1;\n" ::"r"(yes && in ? c.hist + 4u * w : c.spare));
        if (yes && !in && c.hist_g) atomicAdd(c.hist_g + code, 1u);
    } else {
        asm volatile("red.shared.add.u32 [%0], 1;\n" ::"r"(yes ? c.hist + 4u * code : c.spare));
    }
}

}  // namespace
}  // namespace gi
