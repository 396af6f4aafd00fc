// Quality report of a compression (Sec. IV-D, Fig. 4 and the PSNR comparison
// that follows it): statistics of the quant-code histogram (Shannon entropy
// in bits per point, the rate an entropy coder approaches; the number of
// nonzero quant-codes, i.e. points whose prediction error exceeded the bound)
// and the reconstruction error (sum of squares, maximum, PSNR over the value
// range).  Not part of the compression path; used to report what the codes
// and reconstructions of a run look like.
#include <cfloat>

#include "common.cuh"

namespace gi {
namespace {

constexpr int EQ_THREADS = 512;
constexpr int EQ_MAX_BLOCKS = 1024;

struct ErrPartial {
    double sse, maxerr;
    float lo, hi;
    unsigned long long finite;
};

// One block over the 2R bins: counts, entropy (double, bins in ascending order
// per thread, then a fixed tree), largest |q| among kept codes.
__device__ void hist_stats(const uint32_t *__restrict__ hist, int radius, interp_quality *out, int has_err)
{
    __shared__ double s_plogp[EQ_THREADS / 32];
    __shared__ unsigned long long s_n[EQ_THREADS / 32], s_nz[EQ_THREADS / 32];
    __shared__ int s_maxq[EQ_THREADS / 32];
    __shared__ unsigned long long n_total;
    const int bins = 2 * radius;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // pass 1: totals
    unsigned long long n = 0, nz = 0;
    int maxq = 0;
    for (int c = threadIdx.x; c < bins; c += EQ_THREADS) {
        const uint32_t h = hist[c];
        n += h;
        if (c != radius) nz += h;  // nonzero quant-codes, outliers included
        if (h && c != 0 && c != radius) maxq = max(maxq, abs(c - radius));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        n += __shfl_xor_sync(0xffffffffu, n, off);
        nz += __shfl_xor_sync(0xffffffffu, nz, off);
        maxq = max(maxq, __shfl_xor_sync(0xffffffffu, maxq, off));
    }
    if (lane == 0) {
        s_n[warp] = n;
        s_nz[warp] = nz;
        s_maxq[warp] = maxq;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long tn = 0, tz = 0;
        int tq = 0;
        for (int w = 0; w < EQ_THREADS / 32; ++w) {
            tn += s_n[w];
            tz += s_nz[w];
            tq = max(tq, s_maxq[w]);
        }
        n_total = tn;
        out->n = tn;
        out->n_outliers = hist[0];
        out->n_nonzero = tz;
        out->max_abs_q = tq;
        out->reserved = 0;
        if (!has_err) {
            out->n_finite = 0;
            out->sse = out->max_abs_err = out->vmin = out->vmax = out->psnr_db = nan("");
        }
    }
    __syncthreads();
    // pass 2: entropy H = -sum p log2 p, p = h / n
    const double inv_n = n_total ? 1.0 / (double)n_total : 0.0;
    double acc = 0.0;
    for (int c = threadIdx.x; c < bins; c += EQ_THREADS) {
        const uint32_t h = hist[c];
        if (h) {
            const double p = (double)h * inv_n;
            acc -= p * log2(p);
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) s_plogp[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < EQ_THREADS / 32; ++w) t += s_plogp[w];
        out->entropy_bits = t;
    }
}

// Sums of (a - b)^2 that lose nothing against double sums, without double arithmetic per
// point (fp64 runs at 1/64 of the fp32 rate here; five fp64 operations a point bound this
// kernel at 0.77 ms for 384^3 points).  The difference is an exact pair of floats dh + dl
// (Knuth's two-sum); its square, dh^2 + 2 dh dl + dl^2, is taken apart into floats whose
// sum is exact to 2^-70 of it (a product and its fused multiply-add residual); and the
// running sum is a chain of three floats, each taking the rounding errors of the one before
// it, which holds 64 points to about 2^-64 of their sum (2^-52 in the worst case, where
// double additions have 2^-47).  Then it goes into a double.  384^3 points: 881 -> 213 us;
// on sums of 3e6 points 1e-16 off the exact sum, where sums in doubles were 3e-16 .. 8e-16.
// (A chain of two floats took 179 us and was 2^-48 off on single points.)
// A difference whose square would leave the exact range goes straight to the double.  The
// maximum is kept as a pair too (rounding the pair to double gives what rounding the
// difference would).
struct ErrSum {
    double sse, maxerr;
    float s0, s1, s2;  // pending part of the sum
    float mhi, mlo;    // largest |difference| so far as an exact pair
    float vmin, vmax;
    unsigned long long bad;  // non-finite points of x (stored exactly, not counted)
};

__device__ __forceinline__ void err_flush(ErrSum &s)
{
    s.sse += ((double)s.s0 + (double)s.s1) + (double)s.s2;
    s.s0 = s.s1 = s.s2 = 0.0f;
}

// Non-finite points, and differences whose square would leave the exact range.
__device__ __forceinline__ void err_rare(ErrSum &s, float a, float b)
{
    if (!(fabsf(a) <= FLT_MAX)) {
        ++s.bad;
        return;
    }
    s.vmin = fminf(s.vmin, a);
    s.vmax = fmaxf(s.vmax, a);
    const double d = (double)a - (double)b;
    s.sse += d * d;
    s.maxerr = fmax(s.maxerr, fabs(d));
}

// s + v: the sum in s, its rounding error returned (Knuth's two-sum).
__device__ __forceinline__ float add_exact(float &s, float v)
{
    const float t = s + v, q = t - s;
    const float r = (s - (t - q)) + (v - q);
    s = t;
    return r;
}

__device__ __forceinline__ void err_point(ErrSum &s, float a, float b)
{
    float dh = a;
    float dl = add_exact(dh, -b);  // a - b = dh + dl exactly
    const float ad = fabsf(dh);
    // squares of 2^-48 .. 2^55, and of 0, keep every bit of the pair (infinities and NaN fail)
    if (!((ad >= 3.552713678800501e-15f || ad == 0.0f) && ad <= 3.602879701896397e16f)) {
        err_rare(s, a, b);
        return;
    }
    s.vmin = fminf(s.vmin, a);
    s.vmax = fmaxf(s.vmax, a);
    const float p = dh * dh, pe = __fmaf_rn(dh, dh, -p);
    const float d2 = 2.0f * dh, c = d2 * dl, ce = __fmaf_rn(d2, dl, -c);
    // what is left of each addition is at most 2^-24 of it: s2 may round
    const float r0 = add_exact(s.s0, p);
    const float r1 = add_exact(s.s1, r0), r2 = add_exact(s.s1, pe), r3 = add_exact(s.s1, c);
    s.s2 += ((r1 + r2) + r3) + __fmaf_rn(dl, dl, ce);
    // |a - b| = ad + dl with dh's sign taken off
    dl = __uint_as_float(__float_as_uint(dl) ^ (__float_as_uint(dh) & 0x80000000u));
    const bool more = ad > s.mhi || (ad == s.mhi && dl > s.mlo);
    s.mhi = more ? ad : s.mhi;
    s.mlo = more ? dl : s.mlo;
}

__device__ __forceinline__ ErrPartial fold(ErrPartial a, const ErrPartial &b)
{
    a.sse += b.sse;
    a.maxerr = fmax(a.maxerr, b.maxerr);
    a.lo = fminf(a.lo, b.lo);
    a.hi = fmaxf(a.hi, b.hi);
    a.finite += b.finite;
    return a;
}

// Block reduction in a fixed order; thread 0 holds the result.
__device__ ErrPartial block_fold(ErrPartial p)
{
    __shared__ ErrPartial wp[EQ_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        ErrPartial o;
        o.sse = __shfl_down_sync(0xffffffffu, p.sse, off);
        o.maxerr = __shfl_down_sync(0xffffffffu, p.maxerr, off);
        o.lo = __shfl_down_sync(0xffffffffu, p.lo, off);
        o.hi = __shfl_down_sync(0xffffffffu, p.hi, off);
        o.finite = __shfl_down_sync(0xffffffffu, p.finite, off);
        p = fold(p, o);
    }
    __syncthreads();
    if (lane == 0) wp[warp] = p;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < EQ_THREADS / 32; ++w) p = fold(p, wp[w]);
    return p;
}

// The report: block 0 takes the histogram, the others the reconstruction error over the
// finite points of x (grid-stride, 16-byte loads where both fields allow them); the last
// of them folds the partials, in a fixed order, and writes the error statistics.
__global__ void __launch_bounds__(EQ_THREADS, 2) k_quality(const uint32_t *__restrict__ hist, int radius,
                                                        const float *__restrict__ x, const float *__restrict__ xr,
                                                        unsigned long long n, int vec, ErrPartial *partials,
                                                        unsigned int *counter, interp_quality *out)
{
    if (blockIdx.x == 0) {
        hist_stats(hist, radius, out, x != nullptr);
        return;
    }
    const unsigned b = blockIdx.x - 1, nb = gridDim.x - 1;
    const unsigned long long tid = (unsigned long long)b * EQ_THREADS + threadIdx.x;
    const unsigned long long nth = (unsigned long long)nb * EQ_THREADS;
    ErrSum s{0.0, 0.0, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, INFINITY, -INFINITY, 0ull};
    unsigned long long points = 0, done = 0;
    if (vec) {
        const float4 *x4 = reinterpret_cast<const float4 *>(x), *r4 = reinterpret_cast<const float4 *>(xr);
        const unsigned long long n4 = n / 4;
        int pending = 0;
        unsigned long long i = tid;
        auto quad = [&](const float4 &v, const float4 &w) {
            err_point(s, v.x, w.x);
            err_point(s, v.y, w.y);
            err_point(s, v.z, w.z);
            err_point(s, v.w, w.w);
        };
        for (; i + nth < n4; i += 2 * nth) {  // four loads in flight
            const float4 a = __ldcs(x4 + i), c = __ldcs(x4 + i + nth);
            const float4 u = __ldcs(r4 + i), w = __ldcs(r4 + i + nth);
            quad(a, u);
            quad(c, w);
            points += 8;
            if (++pending == 8) {
                err_flush(s);
                pending = 0;
            }
        }
        if (i < n4) {
            quad(__ldcs(x4 + i), __ldcs(r4 + i));
            points += 4;
        }
        err_flush(s);
        done = n4 * 4;
    }
    int pending = 0;
    unsigned long long i = done + tid;
    for (; i < n && i + 3 * nth < n; i += 4 * nth) {  // eight loads in flight
        float a[4], b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            a[j] = __ldcs(x + i + j * nth);
            b[j] = __ldcs(xr + i + j * nth);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) err_point(s, a[j], b[j]);
        points += 4;
        if (++pending == 16) {
            err_flush(s);
            pending = 0;
        }
    }
    for (; i < n; i += nth) {  // three at most
        err_point(s, __ldg(x + i), __ldg(xr + i));
        ++points;
    }
    err_flush(s);
    __shared__ bool last;
    const ErrPartial p = block_fold(ErrPartial{s.sse, fmax(s.maxerr, (double)s.mhi + (double)s.mlo), s.vmin, s.vmax, points - s.bad});
    if (threadIdx.x == 0) {
        partials[b] = p;
        __threadfence();
        last = atomicAdd(counter, 1u) == nb - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    ErrPartial t{0.0, 0.0, INFINITY, -INFINITY, 0ull};
    for (unsigned k = threadIdx.x; k < nb; k += EQ_THREADS) t = fold(t, partials[k]);
    t = block_fold(t);
    if (threadIdx.x != 0) return;
    out->n_finite = t.finite;
    out->sse = t.sse;
    out->max_abs_err = t.maxerr;
    out->vmin = t.finite ? t.lo : nan("");
    out->vmax = t.finite ? t.hi : nan("");
    const double range = (double)t.hi - (double)t.lo;
    out->psnr_db = (t.finite && t.sse > 0.0) ? 20.0 * log10(range) - 10.0 * log10(t.sse / (double)t.finite)
                                             : (t.finite ? INFINITY : nan(""));
    *counter = 0u;
}

}  // namespace

size_t quality_workspace_bytes() { return 256 + sizeof(ErrPartial) * EQ_MAX_BLOCKS; }

cudaError_t launch_quality(const uint32_t *hist, int radius, const float *x, const float *xr, uint64_t n,
                           interp_quality *out, void *ws, cudaStream_t s)
{
    if (!(x && xr && n > 0)) {  // the histogram alone
        k_quality<<<1, EQ_THREADS, 0, s>>>(hist, radius, nullptr, nullptr, 0ull, 0, nullptr, nullptr, out);
        return cudaGetLastError();
    }
    unsigned char *w = static_cast<unsigned char *>(ws);
    unsigned int *counter = reinterpret_cast<unsigned int *>(w);
    const cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    const int vec = aligned16(x) && aligned16(xr);
    unsigned long long blocks = (n + EQ_THREADS * 16ull - 1) / (EQ_THREADS * 16ull);
    const unsigned long long cap = (unsigned long long)min(EQ_MAX_BLOCKS, 2 * sm_count() - 1);  // one wave with block 0
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    k_quality<<<(unsigned)blocks + 1, EQ_THREADS, 0, s>>>(hist, radius, x, xr, (unsigned long long)n, vec,
                                                         reinterpret_cast<ErrPartial *>(w + 256), counter, out);
    return cudaGetLastError();
}

}  // namespace gi
