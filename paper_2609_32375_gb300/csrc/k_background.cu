// k_background.cu -- local background and noise map (paper Section 3.1).
//
//  k_boxstats_u16  one CTA per mesh box: the box's uint16 values go into an
//                  exact 65,536-bin shared-memory histogram (two 16-bit
//                  counters per 32-bit word), summarised into 256 coarse bins
//                  with exact integer count / sum / sum-of-squares prefixes.
//                  The k-sigma clip then runs on the histogram, not on the
//                  pixels: each pass is two range sums and one or two order
//                  statistics, all in exact integer arithmetic.
//  k_boxstats_f32  one CTA per box (<= 16,384 pixels): values in registers,
//                  the clipped set is a range of values, its median from
//                  histograms of the range, sums in compensated FP32.
//  k_mesh_all      boxes with < 50 % good pixels filled from valid neighbours,
//                  both meshes median-filtered, second-derivative tables of the
//                  tensor-product natural spline through the box centres: a
//                  CTA a map, for meshes that fit its shared memory.
//  k_mesh_fill, k_mesh_median, k_spline_lines
//                  the same for larger meshes (FP64 tridiagonal solves).
//  k_bkg_maps      optional full-resolution B(p), sigma(p) output.
#include <float.h>
#include <math.h>

#include "block_select.cuh"
#include "gp_internal.cuh"
#include "gp_launch.h"

namespace gp {

// The box statistics of the clipped set, from which background and rms
// follow.  bkg = median if sigma == 0 or |mean - median| / sigma > 0.3, else
// the mode estimate 2.5 median - 1.5 mean; rms = sigma.
__device__ __forceinline__ void box_result(double med, double mean, double sd, double* bkg, double* rms)
{
    double b;
    if (sd == 0.0 || fabs(mean - med) > 0.3 * sd)
        b = med;
    else
        b = 2.5 * med - 1.5 * mean;
    *bkg = b;
    *rms = sd;
}

// float-float helpers: |a| >= |b| in df_fast; quotients and roots are a float
// estimate and one correction from the exact residual (about 46 bits)
__device__ __forceinline__ DF df_fast(float a, float b)
{
    DF r;
    r.hi = a + b;
    r.lo = b - (r.hi - a);
    return r;
}
__device__ __forceinline__ DF df_div(DF a, float n)
{
    const float q = a.hi / n;
    const float r = fmaf(-q, n, a.hi) + a.lo;
    return df_fast(q, r / n);
}
__device__ __forceinline__ DF df_sqrt(DF a)
{
    if (!(a.hi > 0.f)) return df_zero();
    const float s = sqrtf(a.hi);
    return df_fast(s, (fmaf(-s, s, a.hi) + a.lo) / (2.f * s));
}
// the smallest float >= a (sign = 1), the largest <= a (sign = -1)
__device__ __forceinline__ float df_bound(DF a, float sign)
{
    return a.lo * sign > 0.f ? nextafterf(a.hi, sign * INFINITY) : a.hi;
}
// med + f sd
__device__ __forceinline__ DF df_step(DF med, float f, DF sd)
{
    DF r = med;
    df_add_prod(r, f, sd.hi);
    r.lo = fmaf(f, sd.lo, r.lo);
    return df_fast(r.hi, r.lo);
}
// a 64-bit integer to 48 bits
__device__ __forceinline__ DF df_from(unsigned long long v)
{
    const float hi = __ull2float_rz(v);
    return df_fast(hi, __ull2float_rn(v - (unsigned long long)hi));
}

// ============================================================ uint16 box ===
constexpr int U16_NT = 1024;
constexpr int U16_WORDS = 32768;   // 65,536 16-bit counters

struct HistSums {
    unsigned long long c, s1, s2;
};

// count / sum / sum of squares of the values < v (exact integers)
// executed by one full warp; every lane returns the result
__device__ HistSums hist_prefix(const uint32_t* hist, const unsigned long long* pc, const unsigned long long* ps1,
                                const unsigned long long* ps2, uint32_t v)
{
    const int lane = threadIdx.x & 31;
    uint32_t cb = v >> 8;            // coarse bin of v (256 means "all")
    HistSums r;
    r.c = pc[cb]; r.s1 = ps1[cb]; r.s2 = ps2[cb];
    if (cb >= 256) return r;
    // fine part: values cb*256 .. v-1; lane covers 8 values (4 words)
    unsigned long long c = 0, s1 = 0, s2 = 0;
    uint32_t base = (cb << 8) + (uint32_t)lane * 8u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t w = hist[(base >> 1) + q];
        uint32_t v0 = base + 2u * q, v1 = v0 + 1u;
        uint32_t n0 = w & 0xffffu, n1 = w >> 16;
        if (v0 < v) { c += n0; s1 += (unsigned long long)n0 * v0; s2 += (unsigned long long)n0 * v0 * v0; }
        if (v1 < v) { c += n1; s1 += (unsigned long long)n1 * v1; s2 += (unsigned long long)n1 * v1 * v1; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_xor_sync(0xffffffffu, c, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    r.c += c; r.s1 += s1; r.s2 += s2;
    return r;
}

// the value of global rank r (0-based, r < total count); one full warp
__device__ uint32_t hist_select(const uint32_t* hist, const unsigned long long* pc, unsigned long long r)
{
    const int lane = threadIdx.x & 31;
    // coarse bin: largest cb with pc[cb] <= r  (pc is non-decreasing, pc[0] = 0)
    // lane l checks bins 8l .. 8l+7
    int best = -1;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        int cb = lane * 8 + q;
        if (pc[cb] <= r && pc[cb + 1] > r) best = cb;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    int cb = best < 0 ? 255 : best;
    unsigned long long rem = r - pc[cb];
    // fine: inclusive scan over this coarse bin's 256 counters, 8 per lane
    uint32_t base = ((uint32_t)cb << 8) + (uint32_t)lane * 8u;
    uint32_t cnt[8];
    uint32_t tot = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t w = hist[(base >> 1) + q];
        cnt[2 * q] = w & 0xffffu;
        cnt[2 * q + 1] = w >> 16;
        tot += cnt[2 * q] + cnt[2 * q + 1];
    }
    uint32_t incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    uint32_t excl = incl - tot;
    // the lane whose range holds rem
    bool mine = (excl <= rem) && (rem < incl);
    uint32_t ans = 0;
    if (mine) {
        uint32_t acc = excl;
        for (int q = 0; q < 8; ++q) {
            acc += cnt[q];
            if (rem < acc) { ans = base + q; break; }
        }
    }
    unsigned ball = __ballot_sync(0xffffffffu, mine);
    int src = ball ? (__ffs(ball) - 1) : 0;
    return __shfl_sync(0xffffffffu, ans, src);
}

// queries on the full 65,536-bin histogram
struct FullHist {
    const uint32_t* hist;
    const unsigned long long *pc, *ps1, *ps2;
    bool failed = false;
    __device__ HistSums prefix(uint32_t v) { return hist_prefix(hist, pc, ps1, ps2, v); }
    __device__ uint32_t select(unsigned long long r) { return hist_select(hist, pc, r); }
};

// The integer bounds [x, y] of med -/+ k sigma in float64, with sigma =
// sqrt(num) / n (out of line: few boxes need it)
__device__ __noinline__ uint2 clip_bounds_f64(uint32_t m0, uint32_t m1, unsigned long long num, unsigned long long n,
                                              double k, uint32_t a, uint32_t b)
{
    const double med = 0.5 * ((double)m0 + (double)m1);
    const double sd = sqrt_pos((double)num) * recip_pos((double)n);
    const double ca = ceil(med - k * sd), cb = floor(med + k * sd);
    return make_uint2(ca <= (double)a ? a : (uint32_t)ca, cb >= (double)b ? b : (cb < 0 ? 0u : (uint32_t)cb));
}

// Iterative k-sigma clip about the median on a histogram (one full warp):
// the kept set is always the values in an integer range [a, b]; statistics
// from exact integer sums, median by rank selection.  A float64 warp
// instruction holds this GPU's SM for 16 cycles, and the chain of a pass held
// some 30, so a pass first takes its bounds in float-float, whose error is
// below 2^-44 of their terms.  Only the integer beyond a bound matters: unless
// an integer lies within 2^-40 of the bound (a tie, as two-valued boxes make
// them), float64 would name the same one; then float64 decides.  The final
// statistics are float64.
template <class Q>
__device__ __forceinline__ void clip_histogram(Q& q, uint32_t vmin, uint32_t vmax, double k, int maxiter, double* med_o,
                                               double* mean_o, double* sd_o)
{
    const float kf = (float)k;                // clip_k is a float
    uint32_t a = vmin, b = vmax, m0, m1;
    HistSums lo = q.prefix(a);
    HistSums hi = q.prefix(b + 1u);
    unsigned long long n = hi.c - lo.c, S1 = hi.s1 - lo.s1, S2 = hi.s2 - lo.s2;
    for (int it = 0;; ++it) {
        m0 = q.select(lo.c + (n - 1) / 2);
        m1 = (n & 1ull) ? m0 : q.select(lo.c + n / 2);
        if (it >= maxiter) break;
        // med -/+ k sigma, with sigma = sqrt(n S2 - S1^2) / n
        const unsigned long long num = n * S2 - S1 * S1;
        const DF sd = df_div(df_sqrt(df_from(num)), (float)n);
        DF med;
        med.hi = 0.5f * ((float)m0 + (float)m1);    // exact
        med.lo = 0.f;
        const DF fl = df_step(med, -kf, sd), fh = df_step(med, kf, sd);
        const float tol = 0x1p-40f * fmaf(kf, sd.hi, med.hi);
        const float dl = (fl.hi - rintf(fl.hi)) + fl.lo, dh = (fh.hi - rintf(fh.hi)) + fh.lo;
        uint32_t na, nbv;
        if (fabsf(dl) > tol && fabsf(dh) > tol) {
            float ca = ceilf(fl.hi), cb = floorf(fh.hi);
            if (ca == fl.hi && fl.lo > 0.f) ca += 1.f;
            if (cb == fh.hi && fh.lo < 0.f) cb -= 1.f;
            na = ca <= (float)a ? a : (uint32_t)ca;
            nbv = cb >= (float)b ? b : (cb < 0.f ? 0u : (uint32_t)cb);
        } else {
            const uint2 r = clip_bounds_f64(m0, m1, num, n, k, a, b);
            na = r.x;
            nbv = r.y;
        }
        // At clip_k = 1 the bounds of a two-valued box lie on its values, and
        // rounding can put both inside: nothing more is clipped then
        if (nbv < na) break;
        HistSums nlo = q.prefix(na);
        HistSums nhi = q.prefix(nbv + 1u);
        unsigned long long nn = nhi.c - nlo.c;
        if (nn == n || nn == 0 || q.failed) break;   // the kept set did not change (or emptied), or the query failed
        a = na; b = nbv; lo = nlo; hi = nhi;
        n = nn; S1 = nhi.s1 - nlo.s1; S2 = nhi.s2 - nlo.s2;
    }
    const double in = recip_pos((double)n);
    *med_o = 0.5 * ((double)m0 + (double)m1);
    *mean_o = (double)S1 * in;
    // population variance from exact integers: (n S2 - S1^2) / n^2
    *sd_o = sqrt_pos((double)(n * S2 - S1 * S1)) * in;
}

// rank of quantile q of n good values (features for the learned background)
// : floor(q (n - 1) + 1/2) with q = mantissa 2^-e, exact in integers (and
// without this GPU's slow float64)
__device__ __forceinline__ unsigned long long quantile_rank(float q, uint32_t n)
{
    const uint32_t u = __float_as_uint(q);
    const int e = 150 - (int)(u >> 23);
    return ((unsigned long long)((u & 0x7fffffu) | 0x800000u) * (n - 1u) + (1ull << (e - 1))) >> e;
}

__device__ void boxstats_u16_box(const BoxArgs& A, int box, uint32_t* hist);

// One CTA per box (or, with A.fb_list set, a persistent grid over the boxes
// listed there): the full 65,536-bin histogram in shared memory.
__global__ void __launch_bounds__(U16_NT, 1) k_boxstats_u16(const BoxArgs* __restrict__ batch, const __grid_constant__ BoxArgs one)
{
    pdl_wait();
    pdl_release();
    const BoxArgs& A = frame_args(batch, one);
    extern __shared__ uint32_t hist[];                    // U16_WORDS
    const bool listed = A.fb_list != nullptr;
    const int count = listed ? *A.fb_count : A.nbox;
    for (int i = blockIdx.x; i < count; i += gridDim.x) {
        __syncthreads();                                  // the previous box is done with the histogram
        boxstats_u16_box(A, listed ? A.fb_list[i] : i, hist);
    }
}

__device__ void boxstats_u16_box(const BoxArgs& A, int box, uint32_t* hist)
{
    const uint16_t* __restrict__ img = static_cast<const uint16_t*>(A.img);
    const int64_t pitch = A.pitch;
    const uint8_t* __restrict__ mask = A.mask;
    const int W = A.W, H = A.H, B = A.B, Mx = A.Mx, nbox = A.nbox;
    const double k = A.k;
    const int maxiter = A.maxiter;
    double* __restrict__ bkg_out = A.bkg;
    double* __restrict__ rms_out = A.rms;
    int* __restrict__ valid_out = A.valid;
    float* __restrict__ quant_out = A.quant;
    __shared__ unsigned long long pc[257], ps1[257], ps2[257];
    __shared__ unsigned long long cc_s[256], cs1_s[256], cs2_s[256];
    __shared__ uint32_t red_min[32], red_max[32], red_n[32];

    const int bi = box % Mx, bj = box / Mx;
    const int x0 = bi * B, x1 = min(x0 + B, W);
    const int y0 = bj * B, y1 = min(y0 + B, H);
    const int bw = x1 - x0, bh = y1 - y0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    for (int w = tid; w < U16_WORDS; w += U16_NT) hist[w] = 0u;
    __syncthreads();

    uint32_t vmin = 0xffffffffu, vmax = 0u, ngood = 0u;
    // 8-pixel chunks along each row; rows spread over the CTA
    const int cpr = (bw + 7) >> 3;              // chunks per row
    const int nchunks = cpr * bh;
    const bool vec = ((((uintptr_t)img) & 15) == 0) && ((pitch & 7) == 0) && ((x0 & 7) == 0) && ((bw & 7) == 0) &&
                     !mask;
    auto count = [&](uint32_t u) {
        atomicAdd(&hist[u >> 1], (u & 1u) ? 65536u : 1u);
        vmin = min(vmin, u);
        vmax = max(vmax, u);
        ++ngood;
    };
    if (vec) {
        // four 16-byte loads in flight per thread before the histogram updates
        constexpr int U = 4;
        for (int c0 = tid; c0 < nchunks; c0 += U * U16_NT) {
            uint4 q[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const int c = c0 + k * U16_NT;
                if (c < nchunks) {
                    const int ry = c / cpr, rc = c - ry * cpr;
                    q[k] = __ldg(reinterpret_cast<const uint4*>(img + (int64_t)(y0 + ry) * pitch + x0 + rc * 8));
                }
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                if (c0 + k * U16_NT >= nchunks) break;
                const uint32_t w4[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    count(w4[e] & 0xffffu);
                    count(w4[e] >> 16);
                }
            }
        }
    } else {
        for (int c = tid; c < nchunks; c += U16_NT) {
            const int ry = c / cpr, rc = c - ry * cpr;
            const int y = y0 + ry, xs = x0 + rc * 8;
            const uint16_t* row = img + (int64_t)y * pitch;
            const int nv = min(8, x1 - xs);
            for (int e = 0; e < nv; ++e) {
                if (mask && mask[(int64_t)y * W + xs + e]) continue;
                count(__ldg(row + xs + e));
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        vmin = min(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
        vmax = max(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        ngood += __shfl_xor_sync(0xffffffffu, ngood, o);
    }
    if (lane == 0) { red_min[warp] = vmin; red_max[warp] = vmax; red_n[warp] = ngood; }
    __syncthreads();
    if (warp == 0) {
        vmin = red_min[lane]; vmax = red_max[lane]; ngood = red_n[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            vmin = min(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
            vmax = max(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
            ngood += __shfl_xor_sync(0xffffffffu, ngood, o);
        }
        if (lane == 0) { red_min[0] = vmin; red_max[0] = vmax; red_n[0] = ngood; }
    }
    __syncthreads();
    vmin = red_min[0]; vmax = red_max[0]; ngood = red_n[0];
    const bool valid = ngood > 0 && 2u * ngood >= (uint32_t)(bw * bh);

    if (ngood == 0 || vmin == vmax) {
        // empty box, or a constant one (the only case where one 16-bit
        // counter could have wrapped): statistics are immediate
        if (tid == 0) {
            double med = ngood ? (double)vmin : 0.0;
            double b, r;
            box_result(med, med, 0.0, &b, &r);
            bkg_out[box] = valid ? b : 0.0;
            rms_out[box] = valid ? r : 0.0;
            valid_out[box] = valid;
            if (quant_out)
                for (int q = 0; q < 5; ++q) quant_out[(int64_t)q * nbox + box] = (float)med;
        }
        return;
    }

    // coarse summaries: 256 bins of 256 values
    for (int cb = warp; cb < 256; cb += U16_NT / 32) {
        unsigned long long c = 0, s1 = 0, s2 = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int widx = cb * 128 + lane + 32 * q;
            uint32_t w = hist[widx];
            uint32_t v0 = (uint32_t)widx * 2u, v1 = v0 + 1u;
            uint32_t n0 = w & 0xffffu, n1 = w >> 16;
            c += n0 + n1;
            s1 += (unsigned long long)n0 * v0 + (unsigned long long)n1 * v1;
            s2 += (unsigned long long)n0 * v0 * v0 + (unsigned long long)n1 * v1 * v1;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            c += __shfl_xor_sync(0xffffffffu, c, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) { cc_s[cb] = c; cs1_s[cb] = s1; cs2_s[cb] = s2; }
    }
    __syncthreads();
    if (warp != 0) return;

    // exclusive prefix over the coarse bins (8 per lane)
    {
        unsigned long long c[8], s1[8], s2[8];
        unsigned long long tc = 0, t1 = 0, t2 = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            c[q] = cc_s[lane * 8 + q]; s1[q] = cs1_s[lane * 8 + q]; s2[q] = cs2_s[lane * 8 + q];
            tc += c[q]; t1 += s1[q]; t2 += s2[q];
        }
        unsigned long long ic = tc, i1 = t1, i2 = t2;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long a = __shfl_up_sync(0xffffffffu, ic, o);
            unsigned long long b = __shfl_up_sync(0xffffffffu, i1, o);
            unsigned long long d = __shfl_up_sync(0xffffffffu, i2, o);
            if (lane >= o) { ic += a; i1 += b; i2 += d; }
        }
        unsigned long long ec = ic - tc, e1 = i1 - t1, e2 = i2 - t2;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            pc[lane * 8 + q] = ec; ps1[lane * 8 + q] = e1; ps2[lane * 8 + q] = e2;
            ec += c[q]; e1 += s1[q]; e2 += s2[q];
        }
        if (lane == 31) { pc[256] = ec; ps1[256] = e1; ps2[256] = e2; }
    }
    __syncwarp();

    FullHist fq{hist, pc, ps1, ps2};
    double med, mean, sd;
    clip_histogram(fq, vmin, vmax, k, maxiter, &med, &mean, &sd);
    if (quant_out) {
        const float qs[5] = {0.10f, 0.25f, 0.50f, 0.75f, 0.90f};
        for (int q = 0; q < 5; ++q) {
            uint32_t v = fq.select(quantile_rank(qs[q], ngood));
            if (lane == 0) quant_out[(int64_t)q * nbox + box] = (float)v;
        }
    }
    if (lane == 0) {
        double bb, rr;
        box_result(med, mean, sd, &bb, &rr);
        bkg_out[box] = valid ? bb : 0.0;
        rms_out[box] = valid ? rr : 0.0;
        valid_out[box] = valid;
    }
}

// =================================================== uint16 box, window ===
// The same statistics from a 4,096-bin histogram of a window [w0, w0 + 4096)
// placed around the median of a sample of the box (every 16th row), plus
// exact count / sum / sum-of-squares aggregates of the good values below and
// above the window.  16 KB of shared memory instead of 128 KB, so several
// boxes run per SM.  The clip and the quantiles need exact per-value counts
// only where they query; a query that falls outside the window (a prefix at
// a value strictly inside (vmin, w0) or (w0 + 4096, vmax], a rank below or
// above it) marks the box, which then goes to the full-histogram kernel.
// Prefixes outside the window are still served when the box has few values
// there, kept in a list: hot pixels and cosmic rays (0.05 % of the pixels up to
// full scale) push the first clip bound of nearly every box of a CCD frame
// past the window, and the full-histogram kernel then took as long as this one
// (33 us beside 31 on a 4 MP frame at mesh 128, 775 beside 426 at 81 MP and
// mesh 64; now 4 beside 26, and 4 beside 483).
// Boxes finished here get bit-identical results: the same integer sums, the
// same ranks, the same clip loop.
//
// Threads a box by the number of boxes: 128 keep 8 boxes an SM in flight; a
// frame with fewer boxes than that takes 256 or 512, as it lasts as long as
// one box (256 boxes of 128 x 128: 31 us with 128 threads, 26 with 512; 512
// boxes of 256 x 256: 51 us with 128 threads, 56 with 512, 39 with 256).  Boxes
// of fewer than 32 values a thread keep the smaller CTAs: 576 to 1,024 boxes of
// 64 x 64 take 27 to 31 us with 128 threads, 27 to 39 with 256 or 512 (a handful
// of them 25 and 23, of 90 x 90 31 and 24).
constexpr int NWIN = 4096;
constexpr int NOUT = 1024;              // values outside the window a box may list
constexpr int WCB = 64;                 // values per coarse bin of the window
constexpr int NWC = NWIN / WCB;         // 64 coarse bins

struct WinHist {
    const uint32_t* win;                        // NWIN counters
    const unsigned long long *pc, *ps1, *ps2;   // NWC + 1 prefixes; [0] = the values below the window
    uint32_t w0, vmin, vmax;
    unsigned long long tc, ts1, ts2;            // all good values
    const uint16_t* out;                        // the nout values outside the window (-1: too many to list)
    int nout;
    bool failed = false;

    // the listed values in [a, b)
    __device__ HistSums listed(uint32_t a, uint32_t b)
    {
        HistSums r;
        r.c = r.s1 = r.s2 = 0;
        for (int i = threadIdx.x & 31; i < nout; i += 32) {
            const unsigned long long x = out[i];
            if (x >= a && x < b) { ++r.c; r.s1 += x; r.s2 += x * x; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            r.c += __shfl_xor_sync(0xffffffffu, r.c, o);
            r.s1 += __shfl_xor_sync(0xffffffffu, r.s1, o);
            r.s2 += __shfl_xor_sync(0xffffffffu, r.s2, o);
        }
        return r;
    }

    __device__ HistSums prefix(uint32_t v)
    {
        const int lane = threadIdx.x & 31;
        HistSums r;
        r.c = r.s1 = r.s2 = 0;
        if (v <= vmin) return r;
        if (v > vmax) { r.c = tc; r.s1 = ts1; r.s2 = ts2; return r; }
        if (v < w0 || v > w0 + NWIN) {
            if (nout < 0) { failed = true; return r; }
            if (v < w0) return listed(0u, v);
            r = listed(w0 + NWIN, v);
            r.c += pc[NWC]; r.s1 += ps1[NWC]; r.s2 += ps2[NWC];
            return r;
        }
        const uint32_t d = v - w0, cb = d / WCB;
        r.c = pc[cb]; r.s1 = ps1[cb]; r.s2 = ps2[cb];
        if (cb >= NWC) return r;
        unsigned long long c = 0, s1 = 0, s2 = 0;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t bin = cb * WCB + 2u * lane + e;
            if (bin < d) {
                const unsigned long long nb = win[bin], x = w0 + bin;
                c += nb; s1 += nb * x; s2 += nb * x * x;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            c += __shfl_xor_sync(0xffffffffu, c, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        r.c += c; r.s1 += s1; r.s2 += s2;
        return r;
    }

    __device__ uint32_t select(unsigned long long r)
    {
        const int lane = threadIdx.x & 31;
        if (r < pc[0] || r >= pc[NWC]) { failed = true; return w0; }
        int best = -1;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int cb = 2 * lane + e;
            if (pc[cb] <= r && pc[cb + 1] > r) best = cb;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
        const int cb = best < 0 ? NWC - 1 : best;
        const unsigned long long rem = r - pc[cb];
        const uint32_t base = (uint32_t)cb * WCB + 2u * lane;
        const uint32_t n0 = win[base], n1 = win[base + 1];
        const uint32_t tot = n0 + n1;
        uint32_t incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t excl = incl - tot;
        const bool mine = (excl <= rem) && (rem < incl);
        const uint32_t ans = w0 + base + ((rem < (unsigned long long)excl + n0) ? 0u : 1u);
        const unsigned ball = __ballot_sync(0xffffffffu, mine);
        const int src = ball ? (__ffs(ball) - 1) : 0;
        return __shfl_sync(0xffffffffu, ans, src);
    }
};

template <int WB_NT>
__global__ void __launch_bounds__(WB_NT, 1024 / WB_NT) k_boxstats_win(const BoxArgs* __restrict__ batch,
                                                                      const __grid_constant__ BoxArgs one)
{
    pdl_wait();
    pdl_release();
    const BoxArgs& A = frame_args(batch, one);
    const int box = blockIdx.x;
    if (box >= A.nbox) return;
    const uint16_t* __restrict__ img = static_cast<const uint16_t*>(A.img);
    const int64_t pitch = A.pitch;
    const uint8_t* __restrict__ mask = A.mask;
    const int W = A.W, H = A.H, B = A.B, Mx = A.Mx, nbox = A.nbox;
    __shared__ uint32_t win[NWIN];
    __shared__ uint32_t samp[256];
    __shared__ unsigned long long pc[NWC + 1], ps1[NWC + 1], ps2[NWC + 1];
    __shared__ unsigned long long cc_s[NWC], cs1_s[NWC], cs2_s[NWC];
    __shared__ unsigned long long red64[6][WB_NT / 32];
    __shared__ uint32_t red_min[WB_NT / 32], red_max[WB_NT / 32], red_n[WB_NT / 32];
    __shared__ uint32_t s_w0;
    __shared__ uint16_t out[NOUT];
    __shared__ int nout;

    const int bi = box % Mx, bj = box / Mx;
    const int x0 = bi * B, x1 = min(x0 + B, W);
    const int y0 = bj * B, y1 = min(y0 + B, H);
    const int bw = x1 - x0, bh = y1 - y0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cpr = (bw + 7) >> 3;              // 8-pixel chunks per row
    const bool vec = ((((uintptr_t)img) & 15) == 0) && ((pitch & 7) == 0) && ((x0 & 7) == 0) && ((bw & 7) == 0) &&
                     !mask;

    // f(value) for the good pixels of `rows` rows of the box, `step` apart
    // (rows unaligned, or a mask): neighbouring threads take neighbouring
    // pixels, 8 loads of each array in flight
    auto each_pixel = [&](int rows, int step, auto f) {
        const int dr = WB_NT / bw, dc = WB_NT - dr * bw;
        int ry = tid / bw, rx = tid - ry * bw;
        while (ry < rows) {
            constexpr int U = 8;
            uint16_t v[U];
            uint8_t m[U];
            int n = 0;
#pragma unroll
            for (int k = 0; k < U; ++k) {
                if (ry < rows) {
                    const int64_t y = y0 + ry * step;
                    v[k] = __ldg(img + y * pitch + x0 + rx);
                    m[k] = mask ? __ldg(mask + y * W + x0 + rx) : 0;
                    ++n;
                }
                rx += dc;
                ry += dr;
                if (rx >= bw) { rx -= bw; ++ry; }
            }
#pragma unroll
            for (int k = 0; k < U; ++k)
                if (k < n && !m[k]) f(v[k]);
        }
    };

    for (int w = tid; w < NWIN; w += WB_NT) win[w] = 0u;
    for (int i = tid; i < 256; i += WB_NT) samp[i] = 0u;
    if (tid == 0) nout = 0;
    __syncthreads();

    // ---- sample (every 16th row): median coarse value -> window
    {
        const int srow = (bh + 15) >> 4;
        if (vec) {
            for (int c = tid; c < srow * cpr; c += WB_NT) {
                const int ry = (c / cpr) * 16, rc = c - (c / cpr) * cpr;
                const uint4 q = __ldg(reinterpret_cast<const uint4*>(img + (int64_t)(y0 + ry) * pitch + x0 + rc * 8));
                const uint32_t w4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    atomicAdd(&samp[(w4[e] & 0xffffu) >> 8], 1u);
                    atomicAdd(&samp[w4[e] >> 24], 1u);
                }
            }
        } else {
            each_pixel(srow, 16, [&](uint32_t u) { atomicAdd(&samp[u >> 8], 1u); });
        }
    }
    __syncthreads();
    if (warp == 0) {
        // coarse bin holding the sample median (8 bins per lane)
        uint32_t cnt[8], tot = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) { cnt[q] = samp[lane * 8 + q]; tot += cnt[q]; }
        uint32_t incl = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t ns = __shfl_sync(0xffffffffu, incl, 31);
        const uint32_t rank = ns ? (ns - 1) / 2 : 0;
        uint32_t acc = incl - tot;
        int cb = -1;
        for (int q = 0; q < 8; ++q) {
            if (cb < 0 && rank < acc + cnt[q]) cb = lane * 8 + q;
            acc += cnt[q];
        }
        const bool mine = ns && cb >= 0 && (incl - tot) <= rank && rank < incl;
        const unsigned ball = __ballot_sync(0xffffffffu, mine);
        const int mcb = ball ? __shfl_sync(0xffffffffu, cb, __ffs(ball) - 1) : 0;
        if (lane == 0) {
            const int c = mcb * 256 + 128 - NWIN / 2;
            s_w0 = (uint32_t)(c < 0 ? 0 : (c > 65536 - NWIN ? 65536 - NWIN : c));
        }
    }
    __syncthreads();
    const uint32_t w0 = s_w0;

    // ---- window histogram, aggregates outside it, range and count
    uint32_t vmin = 0xffffffffu, vmax = 0u, ngood = 0u;
    uint32_t lc = 0, ls1 = 0, hc = 0, hs1 = 0;
    unsigned long long ls2 = 0, hs2 = 0;
    auto count = [&](uint32_t u) {
        vmin = min(vmin, u);
        vmax = max(vmax, u);
        ++ngood;
        const uint32_t d = u - w0;
        if (d < (uint32_t)NWIN) {
            atomicAdd(&win[d], 1u);
            return;
        }
        const int i = atomicAdd(&nout, 1);
        if (i < NOUT) out[i] = (uint16_t)u;
        if (u < w0) {
            ++lc; ls1 += u; ls2 += (unsigned long long)u * u;
        } else {
            ++hc; hs1 += u; hs2 += (unsigned long long)u * u;
        }
    };
    if (vec) {
        // 16-byte chunks (8 values); a thread's (row, chunk) advance by the
        // fixed step of one pass of the CTA, without a division per chunk.
        // Both values of a 32-bit word inside the window (the common case)
        // cost a subtraction and a shared atomic each; the rest go through
        // count().  The range of the window's values comes from the
        // histogram afterwards, so only values outside it update vmin/vmax.
        constexpr int U = 4;
        const int dr = WB_NT / cpr, dc = WB_NT - dr * cpr;
        int ry = tid / cpr, rc = tid - ry * cpr;
        while (ry < bh) {
            uint4 q[U];
            int nq = 0;
#pragma unroll
            for (int kk = 0; kk < U; ++kk) {
                if (ry < bh) {
                    q[kk] = __ldg(reinterpret_cast<const uint4*>(img + (int64_t)(y0 + ry) * pitch + x0 + rc * 8));
                    ++nq;
                }
                rc += dc;
                ry += dr;
                if (rc >= cpr) { rc -= cpr; ++ry; }
            }
#pragma unroll
            for (int kk = 0; kk < U; ++kk) {
                if (kk >= nq) break;
                const uint32_t w4[4] = {q[kk].x, q[kk].y, q[kk].z, q[kk].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t u0 = w4[e] & 0xffffu, u1 = w4[e] >> 16;
                    const uint32_t d0 = u0 - w0, d1 = u1 - w0;
                    if ((d0 | d1) < (uint32_t)NWIN) {          // NWIN is a power of two
                        atomicAdd(&win[d0], 1u);
                        atomicAdd(&win[d1], 1u);
                    } else {
                        count(u0);
                        count(u1);
                        ngood -= 2u;                           // counted per chunk below
                    }
                }
                ngood += 8u;
            }
        }
        __syncthreads();
        // the smallest and largest value held in the window
        for (int w = tid; w < NWIN; w += WB_NT)
            if (win[w]) {
                vmin = min(vmin, w0 + (uint32_t)w);
                vmax = max(vmax, w0 + (uint32_t)w);
            }
    } else {
        each_pixel(bh, 1, count);
    }
    unsigned long long agg[6] = {lc, ls1, ls2, hc, hs1, hs2};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        vmin = min(vmin, __shfl_xor_sync(0xffffffffu, vmin, o));
        vmax = max(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        ngood += __shfl_xor_sync(0xffffffffu, ngood, o);
#pragma unroll
        for (int j = 0; j < 6; ++j) agg[j] += __shfl_xor_sync(0xffffffffu, agg[j], o);
    }
    if (lane == 0) {
        red_min[warp] = vmin; red_max[warp] = vmax; red_n[warp] = ngood;
#pragma unroll
        for (int j = 0; j < 6; ++j) red64[j][warp] = agg[j];
    }
    __syncthreads();
    vmin = 0xffffffffu; vmax = 0u; ngood = 0u;
#pragma unroll
    for (int j = 0; j < 6; ++j) agg[j] = 0;
    for (int w = 0; w < WB_NT / 32; ++w) {
        vmin = min(vmin, red_min[w]); vmax = max(vmax, red_max[w]); ngood += red_n[w];
#pragma unroll
        for (int j = 0; j < 6; ++j) agg[j] += red64[j][w];
    }
    const bool valid = ngood > 0 && 2u * ngood >= (uint32_t)(bw * bh);
    if (ngood == 0 || vmin == vmax) {
        // empty or constant box: statistics are immediate (as in the full kernel)
        if (tid == 0) {
            double med = ngood ? (double)vmin : 0.0;
            double b, r;
            box_result(med, med, 0.0, &b, &r);
            A.bkg[box] = valid ? b : 0.0;
            A.rms[box] = valid ? r : 0.0;
            A.valid[box] = valid;
            if (A.quant)
                for (int q = 0; q < 5; ++q) A.quant[(int64_t)q * nbox + box] = (float)med;
        }
        return;
    }

    // ---- coarse summaries of the window (64 bins of 64 values).  Within a
    // coarse bin the count n, sum n d and sum n d^2 of the offsets d < 64
    // from its first value fit 32 bits (n <= 65,536); the sums of v and v^2
    // follow from them exactly in 64 bits.
    for (int cb = warp; cb < NWC; cb += WB_NT / 32) {
        uint32_t c = 0, d1 = 0, d2 = 0;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t d = 2u * lane + e, nb = win[cb * WCB + d];
            c += nb; d1 += nb * d; d2 += nb * d * d;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            c += __shfl_xor_sync(0xffffffffu, c, o);
            d1 += __shfl_xor_sync(0xffffffffu, d1, o);
            d2 += __shfl_xor_sync(0xffffffffu, d2, o);
        }
        if (lane == 0) {
            const unsigned long long base = w0 + (uint32_t)cb * WCB;
            cc_s[cb] = c;
            cs1_s[cb] = base * c + d1;
            cs2_s[cb] = base * base * c + 2ull * base * d1 + d2;
        }
    }
    __syncthreads();
    if (warp != 0) return;
    {
        // prefixes over the coarse bins, starting from the values below the window
        unsigned long long c[2], s1[2], s2[2], tc = 0, t1 = 0, t2 = 0;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            c[e] = cc_s[2 * lane + e]; s1[e] = cs1_s[2 * lane + e]; s2[e] = cs2_s[2 * lane + e];
            tc += c[e]; t1 += s1[e]; t2 += s2[e];
        }
        unsigned long long ic = tc, i1 = t1, i2 = t2;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long a0 = __shfl_up_sync(0xffffffffu, ic, o);
            const unsigned long long a1 = __shfl_up_sync(0xffffffffu, i1, o);
            const unsigned long long a2 = __shfl_up_sync(0xffffffffu, i2, o);
            if (lane >= o) { ic += a0; i1 += a1; i2 += a2; }
        }
        unsigned long long ec = agg[0] + ic - tc, e1 = agg[1] + i1 - t1, e2 = agg[2] + i2 - t2;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            pc[2 * lane + e] = ec; ps1[2 * lane + e] = e1; ps2[2 * lane + e] = e2;
            ec += c[e]; e1 += s1[e]; e2 += s2[e];
        }
        if (lane == 31) { pc[NWC] = ec; ps1[NWC] = e1; ps2[NWC] = e2; }
    }
    __syncwarp();
    WinHist wq;
    wq.win = win; wq.pc = pc; wq.ps1 = ps1; wq.ps2 = ps2;
    wq.w0 = w0; wq.vmin = vmin; wq.vmax = vmax;
    wq.out = out; wq.nout = nout <= NOUT ? nout : -1;
    wq.tc = pc[NWC] + agg[3]; wq.ts1 = ps1[NWC] + agg[4]; wq.ts2 = ps2[NWC] + agg[5];
    double med, mean, sd;
    clip_histogram(wq, vmin, vmax, A.k, A.maxiter, &med, &mean, &sd);
    float qv[5];
    if (A.quant && !wq.failed) {
        const float qs[5] = {0.10f, 0.25f, 0.50f, 0.75f, 0.90f};
        for (int q = 0; q < 5; ++q) qv[q] = (float)wq.select(quantile_rank(qs[q], ngood));
    }
    if (lane != 0) return;
    if (wq.failed) {
        A.fb_list[atomicAdd(A.fb_count, 1)] = box;
        return;
    }
    if (A.quant)
        for (int q = 0; q < 5; ++q) A.quant[(int64_t)q * nbox + box] = qv[q];
    double bb, rr;
    box_result(med, mean, sd, &bb, &rr);
    A.bkg[box] = valid ? bb : 0.0;
    A.rms[box] = valid ? rr : 0.0;
    A.valid[box] = valid;
}

// ============================================================ float32 box ===
// One CTA per box, its values in registers (VPT a thread, NaN where bad or
// clipped away: no range test accepts those).  A clip pass needs the count,
// the sums and the median of the values in a range, so nothing is sorted: a
// histogram of the range, kept as prefix counts, names the few values among
// which the median lies, and later passes (their ranges are nested) use the
// same histogram until their range is an eighth of its own.
//   each pass: values out of range dropped, count and sum  | barrier
//              warp 0: mean; the median's bin              | barrier
//              squared deviations; that bin's values       | barrier
//              warp 0: sigma, median, next range           | barrier
// Bound by instruction issue and the barriers' latency: 34 us for the 256 boxes
// of a 1 MP frame at mesh 64 and 111 us for a masked 9 MP one, where a bitonic
// sort of each box (78 block-wide steps of 4,096 values) took 183 and 721; the
// quantiles of a 17 MP frame take 91 us against 523.  Two float32 values take one paired operation
// in the compensated sums.  The box's mean and sigma are float64; a pass takes
// its mean to the 48 bits that the deviations can use, and its range in
// float-float where that names the same values as float64 would, on one warp:
// this GPU issues a float64 warp instruction every 16 cycles an SM, and its long
// latency sits in the chain of every pass (float64 means there: 1 MP extraction
// 140 -> 145 us, masked 9 MP 309 -> 319).
constexpr int F32_LIST = 64;      // values among which the median is ranked

template <int NT>
struct F32Box {
    __align__(16) uint32_t pre[SEL_BPT * NT + 4];     // values in the bins before; [NB] the total
    __align__(16) SelShared<NT> sel;
    uint32_t wsum[NT / 32];
    DF red[NT / 32];
    uint32_t cnt[NT / 32];                // kept | dropped below << 16
    uint32_t kmin, kmax;
    uint32_t list[5][F32_LIST], nlist[5];
    // what warp 0 tells the others
    float mh, ml, flo, fhi;               // the mean (high, low part); the kept range
    float blo, bhi;                       // range of the values to rank
    uint32_t m, r;                        // how many they are; the (lower) median's rank among them
    int rebuild;
    uint32_t qbin[5], qm[5], qr[5];
    uint32_t flag[SEL_BPT * NT / 32];     // a bit per bin: holds a quantile
};

// s / n to 48 bits (as a float64 quotient split into two floats), n < 2^15:
// the residual of each partial quotient is exact or a rounding below those bits
__device__ __forceinline__ DF df_mean(DF s, float n)
{
    const DF a = df_fast(s.hi, s.lo);
    const float in = 1.f / n, q = a.hi * in;
    DF r;
    r.hi = fmaf(-q, n, a.hi);
    r.lo = 0.f;
    df_add(r, a.lo);
    const float q1 = r.hi * in, q2 = (fmaf(-q1, n, r.hi) + r.lo) * in;
    DF m = df_fast(q, q1);
    m.lo += q2;
    return m;
}
// sum over the first NW lanes (a power of two), in lane 0 .. NW - 1
template <int NW>
__device__ __forceinline__ DF df_sum_lanes(DF v)
{
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1) {
        DF w;
        w.hi = __shfl_xor_sync(0xffffffffu, v.hi, o);
        w.lo = __shfl_xor_sync(0xffffffffu, v.lo, o);
        v = df_merge(v, w);
    }
    return v;
}

// histogram of the keys in [klo, khi], as prefix counts
template <int NT, class Each>
__device__ __forceinline__ void box_histogram(Each each, uint32_t klo, int shift, F32Box<NT>& S)
{
    constexpr int NB = SEL_BPT * NT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int b = tid; b < NB / 4; b += NT) reinterpret_cast<uint4*>(S.pre)[b] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    each([&](uint32_t k) { atomicAdd(&S.pre[(k - klo) >> shift], 1u); });
    __syncthreads();
    uint32_t c[SEL_BPT], tot = 0;
#pragma unroll
    for (int q = 0; q < SEL_BPT / 4; ++q) {
        const uint4 h = reinterpret_cast<const uint4*>(S.pre)[tid * (SEL_BPT / 4) + q];
        c[4 * q] = h.x; c[4 * q + 1] = h.y; c[4 * q + 2] = h.z; c[4 * q + 3] = h.w;
        tot += h.x + h.y + h.z + h.w;
    }
    uint32_t incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) S.wsum[warp] = incl;
    __syncthreads();
    uint32_t e = incl - tot;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) e += w < warp ? S.wsum[w] : 0u;
    uint32_t o[SEL_BPT];
#pragma unroll
    for (int q = 0; q < SEL_BPT; ++q) {
        o[q] = e;
        e += c[q];
    }
#pragma unroll
    for (int q = 0; q < SEL_BPT / 4; ++q)
        reinterpret_cast<uint4*>(S.pre)[tid * (SEL_BPT / 4) + q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2],
                                                                              o[4 * q + 3]);
    if (tid == NT - 1) S.pre[NB] = e;
    __syncthreads();
}

// the bin that holds rank r: the last one with at most r values before it (one full warp)
template <int NT>
__device__ __forceinline__ int find_bin(const F32Box<NT>& S, uint32_t r)
{
    constexpr int NB = SEL_BPT * NT, ST = NB / 32;
    const int lane = threadIdx.x & 31;
    const int top = 31 - __clz(__ballot_sync(0xffffffffu, S.pre[lane * ST] <= r));
    int best = 0;
#pragma unroll
    for (int q = 0; q < ST / 32; ++q) {
        const unsigned m = __ballot_sync(0xffffffffu, S.pre[top * ST + q * 32 + lane] <= r);
        if (m) best = q * 32 + 31 - __clz(m);
    }
    return top * ST + best;
}

// ranks r and r1 (r or r + 1) of the n values list[0..n) (one full warp; n <= F32_LIST)
__device__ __forceinline__ void rank_list(const uint32_t* list, uint32_t n, uint32_t r, uint32_t r1, uint32_t* k0,
                                          uint32_t* k1)
{
    const int lane = threadIdx.x & 31;
    const uint32_t a = lane < n ? list[lane] : 0xffffffffu, b = lane + 32 < n ? list[lane + 32] : 0xffffffffu;
    uint32_t ra = 0, rb = 0;
    for (uint32_t j = 0; j < n; ++j) {
        const uint32_t v = list[j];
        ra += v < a || (v == a && j < (uint32_t)lane);
        rb += v < b || (v == b && j < (uint32_t)lane + 32);
    }
    const bool ha = lane < n, hb = lane + 32 < n;
    // exactly one lane holds each rank
    *k0 = __reduce_max_sync(0xffffffffu, ha && ra == r ? a : hb && rb == r ? b : 0u);
    *k1 = __reduce_max_sync(0xffffffffu, ha && ra == r1 ? a : hb && rb == r1 ? b : 0u);
}

__device__ __forceinline__ int range_shift(uint32_t klo, uint32_t khi, int lb)
{
    const int bits = 32 - __clz(khi - klo);
    return bits > lb ? bits - lb : 0;
}

// the smallest float >= med - k sigma and the largest <= med + k sigma, in
// float64, with sigma = sqrt(dev / n) (out of line: few passes need it)
__device__ __noinline__ float2 clip_bounds_f32(float med0, float med1, DF dev, uint32_t n, double k)
{
    const double med = 0.5 * ((double)med0 + (double)med1), sd = sqrt(fmax(df_value(dev), 0.0) / (double)n);
    const double lo = med - k * sd, hi = med + k * sd;
    float2 b = make_float2((float)lo, (float)hi);
    if ((double)b.x < lo) b.x = nextafterf(b.x, INFINITY);
    if ((double)b.y > hi) b.y = nextafterf(b.y, -INFINITY);
    return b;
}

template <int NT, int VPT, bool QUANT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_boxstats_f32(const BoxArgs* __restrict__ batch,
                                                     const __grid_constant__ BoxArgs one)
{
    pdl_wait();
    pdl_release();
    constexpr int NB = SEL_BPT * NT, NW = NT / 32;
    constexpr int LB = NB == 4096 ? 12 : NB == 2048 ? 11 : 10;
    static_assert(NB == 1 << LB && NW >= 4 && VPT % 2 == 0, "layout");
    const BoxArgs& A = frame_args(batch, one);
    if ((int)blockIdx.x >= A.nbox) return;
    const float* __restrict__ img = static_cast<const float*>(A.img);
    const int64_t pitch = A.pitch;
    const uint8_t* __restrict__ mask = A.mask;
    const int W = A.W, H = A.H, B = A.B, Mx = A.Mx, nbox = A.nbox;
    const double k = A.k;
    const int maxiter = A.maxiter;
    __shared__ __align__(16) F32Box<NT> S;
    const int box = blockIdx.x;
    const int bi = box % Mx, bj = box / Mx;
    const int x0 = bi * B, x1 = min(x0 + B, W);
    const int y0 = bj * B, y1 = min(y0 + B, H);
    const int bw = x1 - x0, np = bw * (y1 - y0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) { S.kmin = 0xffffffffu; S.kmax = 0u; }
    __syncthreads();
    float v[VPT];
    const int dy = NT / bw, dx = NT - dy * bw;
    {
        const int y = tid / bw, xs = tid - y * bw;
        const float* p = img + (int64_t)(y0 + y) * pitch + x0 + xs;
        const int64_t step = dy * pitch + dx, wrap = pitch - bw;
        int x = xs;
#pragma unroll
        for (int q = 0; q < VPT; ++q) {
            v[q] = tid + q * NT < np ? __ldg(p) : NAN;
            p += step;
            x += dx;
            if (x >= bw) { x -= bw; p += wrap; }
        }
        if (mask) {
            const uint8_t* pm = mask + (int64_t)(y0 + y) * W + x0 + xs;
            const int64_t mstep = (int64_t)dy * W + dx, mwrap = W - bw;
            uint8_t b[VPT];
            x = xs;
#pragma unroll
            for (int q = 0; q < VPT; ++q) {
                b[q] = tid + q * NT < np ? __ldg(pm) : 0;
                pm += mstep;
                x += dx;
                if (x >= bw) { x -= bw; pm += mwrap; }
            }
#pragma unroll
            for (int q = 0; q < VPT; ++q)
                if (b[q]) v[q] = NAN;
        }
#pragma unroll
        for (int q = 0; q < VPT; ++q) v[q] = fabsf(v[q]) < INFINITY ? v[q] : NAN;
    }
    auto each = [&](auto f) {
#pragma unroll
        for (int q = 0; q < VPT; ++q)
            if (v[q] == v[q]) f(key_of(v[q]));
    };
    uint32_t ng = 0, klo = 0xffffffffu, khi = 0u;
    each([&](uint32_t key) {
        ++ng;
        klo = min(klo, key);
        khi = max(khi, key);
    });
    ng = __reduce_add_sync(0xffffffffu, ng);
    klo = __reduce_min_sync(0xffffffffu, klo);
    khi = __reduce_max_sync(0xffffffffu, khi);
    if (lane == 0) {
        atomicMin(&S.kmin, klo);
        atomicMax(&S.kmax, khi);
        S.cnt[warp] = ng;
    }
    __syncthreads();
    ng = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) ng += S.cnt[w];
    klo = S.kmin;
    khi = S.kmax;
    __syncthreads();
    const bool valid = ng > 0 && 2 * ng >= (uint32_t)np;
    if (ng == 0) {
        if (tid == 0) { A.bkg[box] = 0; A.rms[box] = 0; A.valid[box] = 0; }
        if (QUANT && tid < 5) A.quant[(int64_t)tid * nbox + box] = 0.f;
        return;
    }
    int shift = range_shift(klo, khi, LB);
    box_histogram<NT>(each, klo, shift, S);

    if constexpr (QUANT) {
        // the learned background's features; nothing reads the clipped statistics then
        const float qs[5] = {0.10f, 0.25f, 0.50f, 0.75f, 0.90f};
        // once more over the bins from the 10 % to the 90 % point, which outliers made wide
        uint32_t below = 0;
        {
            const uint32_t b0 = find_bin<NT>(S, (uint32_t)quantile_rank(qs[0], ng));
            const uint32_t b1 = find_bin<NT>(S, (uint32_t)quantile_rank(qs[4], ng));
            if (shift > 0 && b1 - b0 < NB / 4) {
                below = S.pre[b0];
                const uint32_t top = klo + (b1 << shift) + ((1u << shift) - 1u);
                khi = min(khi, top);
                klo += b0 << shift;
                shift = range_shift(klo, khi, LB);
                __syncthreads();
                box_histogram<NT>([&](auto f) {
                    each([&](uint32_t key) { if (key >= klo && key <= khi) f(key); });
                }, klo, shift, S);
            }
        }
        if (warp == 0) {
            for (int i = lane; i < NB / 32; i += 32) S.flag[i] = 0u;
            __syncwarp();
            for (int q = 0; q < 5; ++q) {
                const uint32_t r = (uint32_t)quantile_rank(qs[q], ng) - below, b = find_bin<NT>(S, r);
                if (lane == 0) {
                    S.qbin[q] = b;
                    S.qm[q] = S.pre[b + 1] - S.pre[b];
                    S.qr[q] = r - S.pre[b];
                    S.nlist[q] = 0;
                    S.flag[b >> 5] |= 1u << (b & 31);
                }
            }
        }
        __syncthreads();
        // the few values of those bins, each into the lists of its quantiles
        each([&](uint32_t key) {
            if (key < klo || key > khi) return;
            const uint32_t b = (key - klo) >> shift;
            if (!((S.flag[b >> 5] >> (b & 31)) & 1u)) return;
            for (int q = 0; q < 5; ++q)
                if (S.qbin[q] == b) {
                    const uint32_t i = atomicAdd(&S.nlist[q], 1u);
                    if (i < F32_LIST) S.list[q][i] = key;
                }
        });
        __syncthreads();
        for (int q = warp; q < 5; q += NW)
            if (S.qm[q] <= F32_LIST) {
                uint32_t k0, k1;
                rank_list(S.list[q], S.qm[q], S.qr[q], S.qr[q], &k0, &k1);
                if (lane == 0) A.quant[(int64_t)q * nbox + box] = key_value(k0);
            }
        for (int q = 0; q < 5; ++q)
            if (S.qm[q] > F32_LIST) {             // many equal or close values
                const uint32_t lo = klo + (S.qbin[q] << shift);
                const uint32_t key = block_select<NT>(each, lo, min(khi, lo + ((1u << shift) - 1u)), S.qr[q], nullptr,
                                                      S.sel);
                if (tid == 0) A.quant[(int64_t)q * nbox + box] = key_value(key);
            }
        if (tid == 0) A.valid[box] = valid;
        return;
    } else {

    float flo = key_value(klo), fhi = key_value(khi);     // the kept range
    uint32_t n = 0, below = 0;                            // kept values; those dropped below the range
    // of the kept set, in warp 0: sum, the two middle values, sum of squared deviations
    DF sum = df_zero(), dev = df_zero();
    float med0 = 0.f, med1 = 0.f;
    const float kf = (float)k;                            // clip_k is a float
    bool rebuild = false;
    for (int it = 0;; ++it) {
        DF2 s2;
        s2.hi = s2.lo = 0ull;
        uint32_t c = 0;
#pragma unroll
        for (int q = 0; q < VPT; q += 2) {
            float x[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const bool in = v[q + e] >= flo && v[q + e] <= fhi;
                c += (v[q + e] < flo ? 65536u : 0u) + (in ? 1u : 0u);
                x[e] = in ? v[q + e] : 0.f;
                v[q + e] = in ? v[q + e] : NAN;
            }
            df2_add(s2, f2pack(x[0], x[1]));
        }
        DF s = df_sum_lanes<32>(df2_sum(s2));
        c = __reduce_add_sync(0xffffffffu, c);
        if (lane == 0) {
            S.red[warp] = s;
            S.cnt[warp] = c;
        }
        __syncthreads();
        c = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) c += S.cnt[w];
        const uint32_t nn = c & 0xffffu;
        if (it > 0 && (nn == n || nn == 0)) break;        // the kept set did not change (or rounding emptied it)
        n = nn;
        below += c >> 16;
        if (rebuild) {
            klo = key_of(flo);
            khi = key_of(fhi);
            shift = range_shift(klo, khi, LB);
            box_histogram<NT>(each, klo, shift, S);
            below = 0;
        }
        const uint32_t r0 = below + (n - 1) / 2, r1 = below + n / 2;
        if (warp == 0) {
            sum = df_sum_lanes<NW>(S.red[lane < NW ? lane : 0]);
            const DF mean = df_mean(sum, (float)n);
            // the bins from the one with rank r0 to the one with rank r1 (those between are empty)
            const uint32_t b0 = find_bin<NT>(S, r0), b1 = r1 < S.pre[b0 + 1] ? b0 : find_bin<NT>(S, r1);
            if (lane == 0) {
                S.mh = mean.hi;
                S.ml = mean.lo;
                // a bin can reach below the kept range: values dropped there still count in its prefix
                const uint32_t kl = klo + (b0 << shift), kh = klo + (b1 << shift) + ((1u << shift) - 1u);
                S.blo = key_value(kl);
                S.bhi = key_value(min(kh, khi));
                S.m = S.pre[b1 + 1] - S.pre[b0];
                S.r = S.pre[b0] > below ? r0 - S.pre[b0] : r0 - below;
                S.nlist[0] = 0;
            }
        }
        __syncthreads();
        const float mh = S.mh, ml = S.ml;
        const float blo = fmaxf(S.blo, flo), bhi = fminf(S.bhi, fhi);
        const bool listed = S.m <= F32_LIST;
        const unsigned long long mh2 = f2pack(mh, mh), ml2 = f2pack(ml, ml);
        s2.hi = s2.lo = 0ull;
#pragma unroll
        for (int q = 0; q < VPT; q += 2) {
            const unsigned long long d = f2sub(f2sub(f2pack(v[q], v[q + 1]), mh2), ml2);
            const float d0 = v[q] == v[q] ? f2lo(d) : 0.f, d1 = v[q + 1] == v[q + 1] ? f2hi(d) : 0.f;
            const unsigned long long dd = f2pack(d0, d1), p = f2mul(dd, dd);
            const unsigned long long np2 = p ^ 0x8000000080000000ull;
            df2_add(s2, p);
            s2.lo = f2add(s2.lo, f2fma(dd, dd, np2));
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (listed && v[q + e] >= blo && v[q + e] <= bhi) {
                    const uint32_t i = atomicAdd(&S.nlist[0], 1u);
                    if (i < F32_LIST) S.list[0][i] = key_of(v[q + e]);
                }
        }
        s = df_sum_lanes<32>(df2_sum(s2));
        if (lane == 0) S.red[warp] = s;
        __syncthreads();
        uint32_t k0 = 0, k1 = 0;
        if (!listed)                                      // many equal or close values
            k0 = block_select<NT>(each, key_of(blo), key_of(bhi), S.r, r1 > r0 ? &k1 : nullptr, S.sel);
        if (warp == 0) {
            dev = df_sum_lanes<NW>(S.red[lane < NW ? lane : 0]);
            if (listed) rank_list(S.list[0], S.nlist[0], S.r, S.r + (r1 - r0), &k0, &k1);
            med0 = key_value(k0);
            med1 = key_value(r1 == r0 ? k0 : k1);
            DF med = df_zero();
            df_add(med, 0.5f * med0);
            df_add(med, 0.5f * med1);
            const DF sd = df_sqrt(df_div(df_fast(dev.hi, dev.lo), (float)n));
            const DF lo = df_step(med, -kf, sd), hi = df_step(med, kf, sd);
            // the float beyond each bound: its nearest float is lo.hi, lo.lo
            // away.  Within 2^-40 of the terms float64 decides (an error of
            // the float-float bound is below 2^-44 of them).
            const float tol = 0x1p-40f * fmaf(kf, sd.hi, fabsf(med.hi));
            float bl, bh;
            if (fabsf(lo.lo) > tol && fabsf(hi.lo) > tol) {
                bl = df_bound(lo, 1.f);
                bh = df_bound(hi, -1.f);
            } else {
                const float2 b = clip_bounds_f32(med0, med1, dev, n, k);
                bl = b.x;
                bh = b.y;
            }
            if (lane == 0) {
                // values >= med - k sd and <= med + k sd
                const float nlo = fmaxf(flo, bl);
                const float nhi = fminf(fhi, bh);
                S.flo = nlo;
                S.fhi = nhi;
                S.rebuild = nlo <= nhi && shift > 0 && (key_of(nhi) - key_of(nlo)) < (khi - klo) / 8;
            }
        }
        if (it >= maxiter) break;
        __syncthreads();
        flo = S.flo;
        fhi = S.fhi;
        rebuild = S.rebuild != 0;
    }
    if (tid == 0) {
        double bb, rr;
        box_result(0.5 * ((double)med0 + (double)med1), df_value(sum) / (double)n,
                   sqrt(fmax(df_value(dev), 0.0) / (double)n), &bb, &rr);
        A.bkg[box] = valid ? bb : 0.0;
        A.rms[box] = valid ? rr : 0.0;
        A.valid[box] = valid;
    }
    }
}

// ====================================================== mesh finalisation ===
constexpr int MF_NT = 1024;

// Fill boxes with < 50 % good pixels from the mean of their valid
// 8-neighbours (sweep after sweep).  One CTA; most meshes have none to fill
// and end at the first look.  250 x 251 boxes: 11 us, and 15 for the medians
// below (1.55 ms when this one CTA copied, sorted and filtered every box).
__global__ void __launch_bounds__(MF_NT)
k_mesh_fill(double* bkg, double* rms, int* valid, double* tmp_b, double* tmp_r, int* tmp_v, int Mx, int My)
{
    pdl_wait();
    pdl_release();
    const int nb = Mx * My, tid = threadIdx.x;
    int good = 0, bad = 0;
#pragma unroll 8
    for (int b = tid; b < nb; b += MF_NT) {
        const int v = valid[b];
        good |= v;
        bad |= !v;
    }
    const bool any = __syncthreads_or(good), some = __syncthreads_or(bad);
    if (!some) return;
    if (!any) {
        for (int b = tid; b < nb; b += MF_NT) { bkg[b] = 0; rms[b] = 0; valid[b] = 1; }
        return;
    }
    for (int sweep = 0; sweep < Mx + My + 2; ++sweep) {
        bool missing = false;
        for (int b = tid; b < nb; b += MF_NT) {
            tmp_b[b] = bkg[b]; tmp_r[b] = rms[b]; tmp_v[b] = valid[b];
            if (valid[b]) continue;
            int i = b % Mx, j = b / Mx, c = 0;
            double sb = 0, sr = 0;
            for (int dj = -1; dj <= 1; ++dj)
                for (int di = -1; di <= 1; ++di) {
                    int ii = i + di, jj = j + dj;
                    if ((di || dj) && ii >= 0 && ii < Mx && jj >= 0 && jj < My && valid[jj * Mx + ii]) {
                        sb += bkg[jj * Mx + ii];
                        sr += rms[jj * Mx + ii];
                        ++c;
                    }
                }
            if (c) { tmp_b[b] = sb / c; tmp_r[b] = sr / c; tmp_v[b] = 1; }
            else missing = true;
        }
        const bool more = __syncthreads_or(missing);
        for (int b = tid; b < nb; b += MF_NT) { bkg[b] = tmp_b[b]; rms[b] = tmp_r[b]; valid[b] = tmp_v[b]; }
        __syncthreads();
        if (!more) break;
    }
}

// Median filter of both meshes over an fsize x fsize window clipped at the
// mesh edge: a thread per box and map.
__global__ void __launch_bounds__(256) k_mesh_median(const double* __restrict__ bkg, const double* __restrict__ rms, int Mx,
                                                     int My, int fsize, float* __restrict__ bkg_out,
                                                     float* __restrict__ rms_out)
{
    pdl_wait();
    pdl_release();
    const int nb = Mx * My, t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2 * nb) return;
    const int map = t / nb, b = t - map * nb, i = b % Mx, j = b / Mx;
    const double* src = map ? rms : bkg;
    double med;
    if (fsize == 3) {
        // the window in registers (absent cells +inf), sorted by odd-even transposition
        double w[9];
        int c = 0;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int ii = i - 1 + k % 3, jj = j - 1 + k / 3;
            const bool in = ii >= 0 && ii < Mx && jj >= 0 && jj < My;
            w[k] = in ? src[jj * Mx + ii] : (double)INFINITY;
            c += in ? 1 : 0;
        }
#pragma unroll
        for (int pass = 0; pass < 9; ++pass)
#pragma unroll
            for (int q = pass & 1; q + 1 < 9; q += 2) {
                const bool sw = w[q + 1] < w[q];
                const double lo = sw ? w[q + 1] : w[q], hi = sw ? w[q] : w[q + 1];
                w[q] = lo;
                w[q + 1] = hi;
            }
        double m0 = w[0], m1 = w[0];
#pragma unroll
        for (int q = 1; q < 9; ++q) {
            if (q == (c - 1) / 2) m0 = w[q];
            if (q == c / 2) m1 = w[q];
        }
        med = (c & 1) ? m1 : 0.5 * (m0 + m1);
    } else {
        const int h = fsize / 2;
        double win[49];
        int c = 0;
        for (int jj = j - h; jj <= j + h; ++jj)
            for (int ii = i - h; ii <= i + h; ++ii)
                if (ii >= 0 && ii < Mx && jj >= 0 && jj < My) {
                    double v = src[jj * Mx + ii];
                    int p = c++;
                    while (p > 0 && win[p - 1] > v) { win[p] = win[p - 1]; --p; }
                    win[p] = v;
                }
        med = (c & 1) ? win[c / 2] : 0.5 * (win[c / 2 - 1] + win[c / 2]);
    }
    (map ? rms_out : bkg_out)[b] = (float)med;
}

// ============================================================ spline tables ===
// Natural-spline second derivatives along lines of n nodes: the tridiagonal
// system h0 M[r-1] + 2 (h0 + h1) M[r] + h1 M[r+1] = rhs, r = 1 .. n - 2, by
// elimination and back substitution in float64.  Both recursions forget: the
// multiplier of what came before is at most about 0.27 a node, so after 32
// nodes 10^-18 of it is left, and a line is cut into chunks of 64 that start
// 32 nodes early (and end 32 late) with a zero there.  The pivots, which
// depend on the node positions only, settle faster still (0.07 a node): each
// is computed from 24 nodes before it.
// A CTA takes 32 lines (a lane each) and one chunk of them; its other warps
// stage.  Bound by the latency of the 224 dependent steps.  A thread per line
// over the whole line, in global memory, with a division a step took 1.6 ms
// and 1.1 ms a map for the two passes of a 250 x 251 mesh; both maps together
// take 57 and 66 us.
constexpr int SL_CH = 64, SL_OV = 32, SL_N = SL_CH + 2 * SL_OV, SL_NT = 128;
constexpr int SL_MAPS = 8;

struct SplineMaps {
    const float* mesh[SL_MAPS];
    float4* tab[SL_MAPS];
    double *X[SL_MAPS], *Y[SL_MAPS];
};

// FINAL = false: X along each mesh row, Y along each mesh column;
// FINAL = true: XY along each row of Y, then (P, X, Y, XY) as float4.
// Grid: x the tiles (those of the rows first), y the map.
template <bool FINAL>
__global__ void __launch_bounds__(SL_NT) k_spline_lines(const __grid_constant__ SplineMaps maps, Axis ax, Axis ay)
{
    pdl_wait();
    pdl_release();
    __shared__ double v[SL_N][33];
    __shared__ double w[SL_N], ib[SL_N], c[SL_N], ih[SL_N + 1];
    const int Mx = ax.n, My = ay.n, tid = threadIdx.x, lane = tid & 31;
    const float* mesh = maps.mesh[blockIdx.y];
    int tile = blockIdx.x;
    const int rtiles = ((My + 31) / 32) * ((Mx + SL_CH - 1) / SL_CH);
    const bool rows = FINAL || tile < rtiles;
    if (!rows) tile -= rtiles;
    const Axis a = rows ? ax : ay;
    const int n = a.n, nline = rows ? My : Mx, nch = (n + SL_CH - 1) / SL_CH;
    const int l0 = tile / nch * 32, c0 = tile % nch * SL_CH, base = c0 - SL_OV;
    // values of nodes base .. base + SL_N - 1 of the lines
    for (int q = tid; q < SL_N * 32; q += SL_NT) {
        const int k = rows ? q % SL_N : q / 32, l = rows ? q / SL_N : q % 32;
        const int node = base + k, line = l0 + l;
        double x = 0.0;
        if (node >= 0 && node < n && line < nline) {
            const int i = rows ? line * Mx + node : node * Mx + line;
            x = FINAL ? maps.Y[blockIdx.y][i] : (double)mesh[i];
        }
        v[k][l] = x;
    }
    auto pos = [&](int i) -> double { return i == n - 1 ? (double)a.tl : (double)a.t0 + (double)i * (double)a.B; };
    auto width = [&](int i) -> double { return pos(i + 1) - pos(i); };   // node i to i + 1
    for (int k = tid; k < SL_N; k += SL_NT) {
        const int r = base + k;
        if (r < 1 || r > n - 2) continue;
        int s = r - 24 > 1 ? r - 24 : 1;
        double b = 2.0 * (width(s - 1) + width(s)), m = 0.0;
        for (++s; s <= r; ++s) {
            const double h0 = width(s - 1);
            m = h0 / b;
            b = 2.0 * (h0 + width(s)) - m * h0;
        }
        w[k] = m;                 // elimination multiplier (0 for r = 1)
        ib[k] = 1.0 / b;
        c[k] = width(r);
        ih[k] = 1.0 / width(r - 1);
        ih[k + 1] = 1.0 / width(r);     // the same value as the next thread's
    }
    __syncthreads();
    const int lo = base > 1 ? base : 1, hi = base + SL_N - 1 < n - 2 ? base + SL_N - 1 : n - 2;
    if (tid < 32) {
        // the first node of a chunk's overlap has no node before it: its rhs
        // needs one, so the sweep starts a node later there
        const int first = lo == base ? lo + 1 : lo, last = hi == base + SL_N - 1 ? hi - 1 : hi;
        double d = 0.0;
        if (first <= last) {
            double vm = v[first - 1 - base][lane], v0 = v[first - base][lane];
            for (int r = first; r <= last; ++r) {
                const int k = r - base;
                const double vp = v[k + 1][lane];
                const double rhs = 6.0 * ((vp - v0) * ih[k + 1] - (v0 - vm) * ih[k]);
                d = rhs - w[k] * d;
                v[k][lane] = d;
                vm = v0;
                v0 = vp;
            }
            double next = 0.0;
            const int end = c0 > 1 ? c0 : 1;
            for (int r = last; r >= end; --r) {
                const int k = r - base;
                next = (v[k][lane] - c[k] * next) * ib[k];
                v[k][lane] = next;
            }
        }
    }
    __syncthreads();
    for (int q = tid; q < SL_CH * 32; q += SL_NT) {
        const int k = rows ? q % SL_CH : q / 32, l = rows ? q / SL_CH : q % 32;
        const int node = c0 + k, line = l0 + l;
        if (node >= n || line >= nline) continue;
        const double M = node < 1 || node > n - 2 ? 0.0 : v[SL_OV + k][l];
        const int i = rows ? line * Mx + node : node * Mx + line;
        if constexpr (FINAL) {
            maps.tab[blockIdx.y][i] = make_float4(mesh[i], (float)maps.X[blockIdx.y][i], (float)maps.Y[blockIdx.y][i], (float)M);
        } else {
            (rows ? maps.X : maps.Y)[blockIdx.y][i] = M;
        }
    }
}

__global__ void k_bkg_maps(SplineTab sb, SplineTab sr, int W, int H, float* bmap, float* rmap)
{
    const int64_t n = (int64_t)W * H;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
        float x = (float)(p % W), y = (float)(p / W);
        if (bmap) bmap[p] = spline_eval(sb, x, y);
        if (rmap) rmap[p] = spline_eval(sr, x, y);
    }
}

// ====================================================== fused mesh kernel ===
// One CTA a map does the whole mesh stage in shared memory when the mesh has
// at most MESH_SMEM_NODES nodes: invalid-box fill, median filter, and the
// spline tables.  The tridiagonal matrix of the natural spline
// depends only on the node positions, so each axis is factorised once
// (multipliers and reciprocal pivots) and every line is then solved with
// FMAs only.  FP32 throughout: the tables are stored in FP32 anyway, and the
// diagonally dominant spline system loses nothing that matters at 1e-5.
// Bound by latency, a line's recurrences above all: the lines' values are
// loaded SL_AHEAD nodes ahead of them.  A 16 x 16 mesh
// takes 7.5 us and a 48 x 49 one 17.6 (13 and 34 with both maps in one CTA, a
// load before each step and every pivot divided out).
constexpr int MESH_SMEM_NODES = 4096;
constexpr int MA_NT = 1024;

// byte offset of the LU scratch in k_mesh_all's shared memory: three float
// arrays and two int arrays of n entries, rounded up to 16 bytes
__host__ __device__ __forceinline__ size_t mesh_lu_offset(int n)
{
    const size_t end = (size_t)n * (3 * sizeof(float) + 2 * sizeof(int));
    return (end + 15) & ~(size_t)15;
}

struct AxisLU {
    float* w;      // elimination multipliers  (index r = 1..n-2)
    float* ib;     // reciprocal pivots
    float* c;      // super-diagonal
    float* ih;     // 1 / interval width (n-1 entries)
};

__device__ __forceinline__ float node_pos(const Axis& a, int i)
{
    return (i == a.n - 1) ? a.tl : a.t0 + (float)i * a.B;
}

// a warp; the pivots' recurrence on its first lane.  With equal intervals it
// soon repeats its values, and a step whose operands are those of the step
// before has its results.
__device__ void factor_axis(const Axis& a, AxisLU L, int lane)
{
    const int n = a.n;
    for (int i = lane; i + 1 < n; i += 32) L.ih[i] = 1.f / (node_pos(a, i + 1) - node_pos(a, i));
    if (lane) return;
    float bprev = 0.f, cprev = 0.f, h0p = 0.f, h1p = 0.f, bpp = 0.f, w = 0.f, ib = 0.f, b = 0.f;
    for (int r = 1; r <= n - 2; ++r) {
        const float h0 = node_pos(a, r) - node_pos(a, r - 1), h1 = node_pos(a, r + 1) - node_pos(a, r);
        if (!(r > 2 && h0 == h0p && h1 == h1p && bprev == bpp && cprev == h0)) {
            b = 2.f * (h0 + h1);
            w = 0.f;
            if (r > 1) {
                w = h0 / bprev;
                b -= w * cprev;
            }
            ib = 1.f / b;
        }
        L.w[r] = w;
        L.ib[r] = ib;
        L.c[r] = h1;
        h0p = h0;
        h1p = h1;
        bpp = bprev;
        bprev = b;
        cprev = h1;
    }
}

// second derivatives of one line (values v, stride vs) into M (stride ms)
constexpr int SL_AHEAD = 8;
__device__ void solve_line(const AxisLU& L, int n, const float* v, int vs, float* M, int ms)
{
    M[0] = 0.f;
    if (n >= 2) M[(n - 1) * ms] = 0.f;
    if (n < 3) return;
    float dprev = 0.f, vr = v[vs], pr = (vr - v[0]) * L.ih[0];      // slope before node r
    for (int r0 = 1; r0 <= n - 2; r0 += SL_AHEAD) {
        float vn[SL_AHEAD], ih[SL_AHEAD], w[SL_AHEAD], d[SL_AHEAD];
#pragma unroll
        for (int j = 0; j < SL_AHEAD; ++j) {
            const int r = min(r0 + j, n - 2);
            vn[j] = v[(r + 1) * vs];
            ih[j] = L.ih[r];
            w[j] = L.w[r];
        }
#pragma unroll
        for (int j = 0; j < SL_AHEAD; ++j) {
            const float dv = vn[j] - vr;
            d[j] = 6.f * fmaf(dv, ih[j], -pr);
            pr = __fmul_rn(dv, ih[j]);
            vr = vn[j];
        }
#pragma unroll
        for (int j = 0; j < SL_AHEAD; ++j)
            if (r0 + j <= n - 2) {
                dprev = fmaf(-w[j], dprev, d[j]);
                M[(r0 + j) * ms] = dprev;        // forward-eliminated right-hand side
            }
    }
    float next = 0.f;
    for (int r0 = n - 2; r0 >= 1; r0 -= SL_AHEAD) {
        float c[SL_AHEAD], ib[SL_AHEAD], m[SL_AHEAD];
#pragma unroll
        for (int j = 0; j < SL_AHEAD; ++j) {
            const int r = max(r0 - j, 1);
            c[j] = L.c[r];
            ib[j] = L.ib[r];
            m[j] = M[r * ms];
        }
#pragma unroll
        for (int j = 0; j < SL_AHEAD; ++j)
            if (r0 - j >= 1) {
                next = fmaf(-c[j], next, m[j]) * ib[j];
                M[(r0 - j) * ms] = next;
            }
    }
}

// mode 0: raw box statistics -> fill, filter, write meshes, tables
// mode 1: tables only, from the float meshes given in bkg_out / rms_out
// blockIdx.x = the map: background, noise
__global__ void __launch_bounds__(MA_NT) k_mesh_all(const MeshArgs* __restrict__ batch,
                                                    const __grid_constant__ MeshArgs one)
{
    pdl_wait();
    pdl_release();
    const MeshArgs& MA = frame_args(batch, one);
    const double* __restrict__ raw = blockIdx.x ? MA.rms_raw : MA.bkg_raw;
    const int* __restrict__ valid_raw = MA.valid;
    const Axis ax = MA.ax, ay = MA.ay;
    const int fsize = MA.fsize, mode = MA.mode;
    float* out = blockIdx.x ? MA.rms_mesh : MA.bkg_mesh;
    float4* tab = blockIdx.x ? MA.tab_r : MA.tab_b;
    extern __shared__ __align__(16) float sh[];
    unsigned char* sh_bytes = reinterpret_cast<unsigned char*>(sh);
    // shared-memory rows are Ms = Mx | 1 wide (odd), so the row-direction
    // solves, one row per lane, hit 32 different banks
    const int Mx = ax.n, My = ay.n, n = Mx * My, tid = threadIdx.x;
    const int Ms = Mx | 1, ns = Ms * My;
    float* A = sh;             // raw values; X
    float* T = A + ns;         // fill scratch; Y
    float* P = T + ns;         // filtered values; XY
    int* V0 = reinterpret_cast<int*>(P + ns);
    int* V1 = V0 + ns;
    const int nl = Mx > My ? Mx : My;
    // the LU scratch starts at the first 16-byte boundary after V1
    float* lu = reinterpret_cast<float*>(sh_bytes + mesh_lu_offset(ns));
    AxisLU Lx{lu, lu + nl, lu + 2 * nl, lu + 3 * nl};
    AxisLU Ly{lu + 4 * nl, lu + 5 * nl, lu + 6 * nl, lu + 7 * nl};
    // two warps factor the spline systems (first needed by the solves)
    if (tid >= MA_NT - 32) factor_axis(ax, Lx, tid & 31);
    else if (tid >= MA_NT - 64) factor_axis(ay, Ly, tid & 31);

    if (mode == 0) {
        bool good = false, gap = false;
        for (int b = tid; b < n; b += MA_NT) {
            const int sb_ = (b / Mx) * Ms + b % Mx, v = valid_raw[b];
            A[sb_] = (float)raw[b];
            V0[sb_] = v;
            good |= v != 0;
            gap |= v == 0;
        }
        const bool any = __syncthreads_or(good);
        if (!any) {
            for (int i = tid; i < ns; i += MA_NT) A[i] = 0.f;
            __syncthreads();
        }
        bool more = __syncthreads_or(gap) && any;
        // fill invalid boxes from valid 8-neighbours, sweep after sweep
        for (int sweep = 0; more && sweep < Mx + My + 2; ++sweep) {
            bool missing = false;
            for (int b = tid; b < n; b += MA_NT) {
                const int i = b % Mx, j = b / Mx, sb_ = j * Ms + i;
                T[sb_] = A[sb_]; V1[sb_] = V0[sb_];
                if (V0[sb_]) continue;
                int c = 0;
                float sum = 0.f;
                for (int dj = -1; dj <= 1; ++dj)
                    for (int di = -1; di <= 1; ++di) {
                        const int ii = i + di, jj = j + dj;
                        if ((di || dj) && ii >= 0 && ii < Mx && jj >= 0 && jj < My && V0[jj * Ms + ii]) {
                            sum += A[jj * Ms + ii];
                            ++c;
                        }
                    }
                if (c) { T[sb_] = sum / c; V1[sb_] = 1; }
                else missing = true;
            }
            more = __syncthreads_or(missing);
            for (int b = tid; b < n; b += MA_NT) {
                const int sb_ = (b / Mx) * Ms + b % Mx;
                A[sb_] = T[sb_]; V0[sb_] = V1[sb_];
            }
            __syncthreads();
        }
        // median filter (window clipped at the mesh edge) -> float mesh
        const int h = fsize / 2;
        for (int b = tid; b < n && fsize == 3; b += MA_NT) {
            // 3 x 3: the window in registers (absent cells +inf), sorted by
            // odd-even transposition; the same order statistics as below
            const int i = b % Mx, j = b / Mx;
            float w[9];
            int c = 0;
#pragma unroll
            for (int dj = -1; dj <= 1; ++dj)
#pragma unroll
                for (int di = -1; di <= 1; ++di) {
                    const int ii = i + di, jj = j + dj;
                    const bool in = ii >= 0 && ii < Mx && jj >= 0 && jj < My;
                    w[(dj + 1) * 3 + di + 1] = in ? A[jj * Ms + ii] : INFINITY;
                    c += in ? 1 : 0;
                }
#pragma unroll
            for (int pass = 0; pass < 9; ++pass)
#pragma unroll
                for (int q = pass & 1; q + 1 < 9; q += 2) {
                    const float lo = fminf(w[q], w[q + 1]), hi = fmaxf(w[q], w[q + 1]);
                    w[q] = lo;
                    w[q + 1] = hi;
                }
            float m0 = w[0], m1 = w[0];
#pragma unroll
            for (int q = 1; q < 9; ++q) {
                if (q == (c - 1) / 2) m0 = w[q];
                if (q == c / 2) m1 = w[q];
            }
            P[j * Ms + i] = out[b] = (c & 1) ? m1 : 0.5f * (m0 + m1);
        }
        for (int b = tid; b < n && fsize != 3; b += MA_NT) {
            const int i = b % Mx, j = b / Mx;
            float win[49];
            int c = 0;
            for (int jj = j - h; jj <= j + h; ++jj)
                for (int ii = i - h; ii <= i + h; ++ii)
                    if (ii >= 0 && ii < Mx && jj >= 0 && jj < My) {
                        const float v = A[jj * Ms + ii];
                        int p = c++;
                        while (p > 0 && win[p - 1] > v) { win[p] = win[p - 1]; --p; }
                        win[p] = v;
                    }
            P[j * Ms + i] = out[b] = (c & 1) ? win[c / 2] : 0.5f * (win[c / 2 - 1] + win[c / 2]);
        }
    } else {
        for (int b = tid; b < n; b += MA_NT) P[(b / Mx) * Ms + b % Mx] = out[b];
    }
    __syncthreads();
    // spline table: X (rows) and Y (columns) at once, then XY (rows of Y)
    for (int q = tid; q < My + Mx; q += MA_NT) {
        if (q < My) solve_line(Lx, Mx, P + q * Ms, 1, A + q * Ms, 1);
        else solve_line(Ly, My, P + (q - My), Ms, T + (q - My), Ms);
    }
    __syncthreads();
    // the values go out before XY overwrites them
    for (int b = tid; b < n; b += MA_NT) {
        const int sb_ = (b / Mx) * Ms + b % Mx;
        tab[b] = make_float4(P[sb_], A[sb_], T[sb_], 0.f);
    }
    __syncthreads();
    for (int q = tid; q < My; q += MA_NT) solve_line(Lx, Mx, T + q * Ms, 1, P + q * Ms, 1);
    __syncthreads();
    for (int b = tid; b < n; b += MA_NT) tab[b].w = P[(b / Mx) * Ms + b % Mx];
}

size_t mesh_all_smem(int Mx, int My)
{
    const size_t ns = (size_t)(Mx | 1) * My;     // odd row stride (see k_mesh_all)
    const size_t nl = Mx > My ? Mx : My;
    return mesh_lu_offset((int)ns) + 8 * nl * sizeof(float);
}

// Meshes for k_mesh_all, whose splines are solved in float32: up to
// MESH_SMEM_NODES nodes, and no axis so long (some 2,800 nodes and more) that 32
// bytes a node and 32 a node of the longer axis exceed 220 KB.  Those lines
// take the float64 solves of the larger meshes, although k_mesh_all's own
// 20 bytes a node would fit.
bool mesh_fits_smem(int Mx, int My)
{
    const size_t ns = (size_t)(Mx | 1) * My, nl = Mx > My ? Mx : My;
    return (size_t)Mx * My <= (size_t)MESH_SMEM_NODES && (((ns * 32 + 15) & ~(size_t)15) + 32 * nl) <= 220 * 1024;
}

MeshArgs mesh_args(const double* bkg_raw, const double* rms_raw, const int* valid, Axis ax, Axis ay, int fsize,
                   int mode, float* bkg_mesh, float* rms_mesh, float4* tab_b, float4* tab_r)
{
    MeshArgs a;
    a.bkg_raw = bkg_raw; a.rms_raw = rms_raw; a.valid = valid;
    a.ax = ax; a.ay = ay; a.fsize = fsize; a.mode = mode;
    a.bkg_mesh = bkg_mesh; a.rms_mesh = rms_mesh; a.tab_b = tab_b; a.tab_r = tab_r;
    return a;
}

// smem = the largest frame's mesh_all_smem
cudaError_t launch_mesh_all_any(const MeshArgs& one, const MeshArgs* batch, int nframes, size_t smem, cudaStream_t st)
{
    cudaFuncSetAttribute(k_mesh_all, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_dep(k_mesh_all, dim3(2, nframes), dim3(MA_NT), smem, st, batch, one);
    return cudaGetLastError();
}

cudaError_t launch_mesh_all(const double* bkg_raw, const double* rms_raw, const int* valid, Axis ax, Axis ay,
                            int fsize, int mode, float* bkg_mesh, float* rms_mesh, float4* tab_b, float4* tab_r,
                            cudaStream_t st)
{
    const MeshArgs a = mesh_args(bkg_raw, rms_raw, valid, ax, ay, fsize, mode, bkg_mesh, rms_mesh, tab_b, tab_r);
    return launch_mesh_all_any(a, nullptr, 1, mesh_all_smem(ax.n, ay.n), st);
}

// --------------------------------------------------------------- launchers ---
BoxArgs box_args(const Image& im, int B, double k, int maxiter, double* bkg, double* rms, int* valid, float* quant)
{
    BoxArgs a;
    a.img = im.data; a.pitch = im.pitch; a.mask = im.mask;
    a.W = im.W; a.H = im.H; a.B = B;
    a.Mx = (im.W + B - 1) / B;
    a.nbox = a.Mx * ((im.H + B - 1) / B);
    a.k = k; a.maxiter = maxiter;
    a.bkg = bkg; a.rms = rms; a.valid = valid; a.quant = quant;
    a.fb_list = nullptr; a.fb_count = nullptr;
    return a;
}

// one frame (batch == nullptr) or nframes frames whose arguments are in the
// device array batch; maxbox = the largest frame's box count
cudaError_t launch_boxstats_any(const BoxArgs& one, const BoxArgs* batch, int nframes, int maxbox, int is_f32,
                                cudaStream_t st)
{
    dim3 grid(maxbox, nframes);
    if (!is_f32 && one.fb_list) {
        // windowed histograms, then the full histogram for the boxes they
        // could not finish (a persistent grid over the fallback lists)
        const int64_t boxes = (int64_t)maxbox * nframes, area = (int64_t)one.B * one.B;
        if (boxes >= 8 * 152 || area < 256 * 32) launch_dep(k_boxstats_win<128>, grid, dim3(128), 0, st, batch, one);
        else if (boxes >= 2 * 152 || area < 512 * 32) launch_dep(k_boxstats_win<256>, grid, dim3(256), 0, st, batch, one);
        else launch_dep(k_boxstats_win<512>, grid, dim3(512), 0, st, batch, one);
        const size_t smem = U16_WORDS * sizeof(uint32_t);
        cudaFuncSetAttribute(k_boxstats_u16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        launch_dep(k_boxstats_u16, dim3(maxbox < 152 ? maxbox : 152, nframes), dim3(U16_NT), smem, st, batch, one);
        return cudaGetLastError();
    }
    if (!is_f32) {
        const size_t smem = U16_WORDS * sizeof(uint32_t);
        cudaFuncSetAttribute(k_boxstats_u16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_boxstats_u16<<<grid, U16_NT, smem, st>>>(batch, one);
    } else {
        // threads and values a thread by box area (the frames of a batch share B)
        const int area = one.B * one.B;
        auto run = [&](auto kern, auto quant, int nt) {
            launch_dep(one.quant ? quant : kern, grid, dim3(nt), 0, st, batch, one);
        };
        if (area <= 128 * 8) run(k_boxstats_f32<128, 8, false>, k_boxstats_f32<128, 8, true>, 128);
        else if (area <= 256 * 16) run(k_boxstats_f32<256, 16, false>, k_boxstats_f32<256, 16, true>, 256);
        else run(k_boxstats_f32<512, 32, false>, k_boxstats_f32<512, 32, true>, 512);
    }
    return cudaGetLastError();
}

cudaError_t launch_boxstats(const Image& im, int B, double k, int maxiter, double* bkg, double* rms, int* valid,
                            float* quant, cudaStream_t st)
{
    const BoxArgs a = box_args(im, B, k, maxiter, bkg, rms, valid, quant);
    return launch_boxstats_any(a, nullptr, 1, a.nbox, im.is_f32, st);
}

cudaError_t launch_mesh_finalize(double* bkg, double* rms, int* valid, double* tmp_b, double* tmp_r, int* tmp_v,
                                 int Mx, int My, int fsize, float* bkg_out, float* rms_out, cudaStream_t st)
{
    launch_dep(k_mesh_fill, dim3(1), dim3(MF_NT), 0, st, bkg, rms, valid, tmp_b, tmp_r, tmp_v, Mx, My);
    launch_dep(k_mesh_median, dim3((2 * Mx * My + 255) / 256), dim3(256), 0, st, bkg, rms, Mx, My, fsize, bkg_out, rms_out);
    return cudaGetLastError();
}

// tables of nmap meshes (mesh[m] -> tab[m]) on the same axes; scratch as for one
cudaError_t launch_spline_tables(const float* const* mesh, float4* const* tab, int nmap, Axis ax, Axis ay, double* scratch,
                                 int* nlaunch, cudaStream_t st)
{
    const int64_t nn = (int64_t)ax.n * ay.n;
    // X and Y of as many maps at a time as the scratch holds (two at least)
    const int64_t room = (int64_t)spline_scratch_doubles(ax.n, ay.n) / (2 * nn);
    const int most = (int)(room < SL_MAPS ? room : SL_MAPS);
    const int rt = ((ay.n + 31) / 32) * ((ax.n + SL_CH - 1) / SL_CH), ct = ((ax.n + 31) / 32) * ((ay.n + SL_CH - 1) / SL_CH);
    for (int m0 = 0; m0 < nmap; m0 += most) {
        const int k = nmap - m0 < most ? nmap - m0 : most;
        SplineMaps sm = {};
        for (int m = 0; m < k; ++m) {
            sm.mesh[m] = mesh[m0 + m];
            sm.tab[m] = tab[m0 + m];
            sm.X[m] = scratch + 2 * nn * m;
            sm.Y[m] = sm.X[m] + nn;
        }
        launch_dep(k_spline_lines<false>, dim3(rt + ct, k), dim3(SL_NT), 0, st, sm, ax, ay);
        launch_dep(k_spline_lines<true>, dim3(rt, k), dim3(SL_NT), 0, st, sm, ax, ay);
        if (nlaunch) *nlaunch += 2;
    }
    return cudaGetLastError();
}

size_t spline_scratch_doubles(int Mx, int My)
{
    return (size_t)5 * Mx * My + (size_t)2 * (Mx + My) * (Mx + My);
}

cudaError_t launch_bkg_maps(const SplineTab& sb, const SplineTab& sr, int W, int H, float* bmap, float* rmap,
                            cudaStream_t st)
{
    int64_t n = (int64_t)W * H;
    int64_t nb_ = (n + 255) / 256;
    int blocks = (int)(nb_ < 152 * 16 ? nb_ : 152 * 16);
    k_bkg_maps<<<blocks, 256, 0, st>>>(sb, sr, W, H, bmap, rmap);
    return cudaGetLastError();
}

}  // namespace gp
