// k_ropt.cu -- the optimal aperture radius (paper Section 3.4): the radius
// of largest S/N is searched on the growth curves of high-S/N isolated
// calibrators, log10 r_opt = a log10 nu + b is fitted to them (nu the
// detection significance), and every other source takes the radius of the
// fit.
//
//  k_ropt_nu     one warp per catalog row: nu = F / sigma at the row's peak
//                pixel (F the matched filter of m = I - B with the detection
//                kernel, mirror border, bad pixels 0) and the index of the
//                largest S/N = flux / fluxerr of its growth curve (the first
//                on ties; 0 where fluxerr <= 0).
//  k_iso_*       isolation on a grid of cells at least d_iso wide: count,
//                scan, fill, then each row looks for another centroid closer
//                than d_iso in its 3 x 3 cells, and takes the calibrator test;
//                each CTA's calibrators give a part of the fit's centred sums.
//  k_ropt_fit    one CTA: least squares of log10 r on log10 nu over the
//                calibrators from those parts, in a fixed order.
//  k_ropt_assign one thread per row: the calibrators keep their best radius,
//                the others take the grid radius nearest to the fit's
//                (ties to the larger).
#include <math.h>
#include <string.h>

#include <algorithm>

#include "block_select.cuh"
#include "gp_internal.cuh"
#include "gp_launch.h"

namespace gp {

struct RoptTaps {
    int kw, kh;
    float t[KMAX];
};

struct RoptRadii {
    int nr;
    int r[GP_GROWTH_MAX_NR];
};

// A warp per row: a lane computes m under one tap (the float64-free part that
// waits on memory), every lane then adds the taps in their order; the radii's
// S/N come one a lane.  15,000 rows: 32 us with a thread per row, 17 so.
template <bool F32>
__global__ void __launch_bounds__(256) k_ropt_nu(Image im, SplineTab sb, SplineTab sr,
                                                 const __grid_constant__ RoptTaps K, const int* __restrict__ xp,
                                                 const int* __restrict__ yp, const double* __restrict__ flux,
                                                 const double* __restrict__ ferr, int nr, const int* __restrict__ n_dev,
                                                 int cap, float* nu, int* kopt)
{
    const int n = min(*n_dev, cap);
    const int W = im.W, H = im.H, hx = K.kw / 2, hy = K.kh / 2, ntap = K.kw * K.kh;
    const int lane = threadIdx.x & 31;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += (gridDim.x * blockDim.x) >> 5) {
        const int x0 = xp[i], y0 = yp[i];
        float F = 0.f;
        for (int t0 = 0; t0 < ntap; t0 += 32) {
            const int t = t0 + lane;
            float m = 0.f;
            if (t < ntap) {
                const int v = t / K.kw, u = t - v * K.kw;
                const int x = mirror_idx(x0 + u - hx, W), y = mirror_idx(y0 + v - hy, H);
                bool bad;
                const float val = load_px<F32>(im, x, y, bad);
                m = bad ? 0.f : val - spline_eval(sb, (float)x, (float)y);
            }
            const int e = min(32, ntap - t0);
            for (int j = 0; j < e; ++j) F = fmaf(K.t[t0 + j], __shfl_sync(0xffffffffu, m, j), F);
        }
        const float s = spline_eval(sr, (float)x0, (float)y0);
        // the first of the largest S/N (0 where the error is not positive; a
        // NaN in front stays): by float32 quotients where one of them is
        // clear of the others by more than their rounding, else in float64
        double f = 0.0, e = 0.0;
        if (lane < nr) {
            f = flux[(int64_t)i * nr + lane];
            e = ferr[(int64_t)i * nr + lane];
        }
        const float ff = (float)f, ef = (float)e;
        const float qf = lane < nr ? (e > 0.0 ? ff / ef : 0.f) : -INFINITY;
        const float top = key_value(__reduce_max_sync(0xffffffffu, key_of(qf == qf ? qf : INFINITY)));
        const unsigned near = __ballot_sync(0xffffffffu, !(qf < top * (1.f - 1e-6f)));
        int best = __ffs(near) - 1;
        if (!(top > 1e-30f && top < 1e30f) || (near & (near - 1u))) {
            const double q = lane < nr && e > 0.0 ? f / e : 0.0;
            best = 0;
            double bs = __shfl_sync(0xffffffffu, q, 0);
            for (int k = 1; k < nr; ++k) {
                const double o = __shfl_sync(0xffffffffu, q, k);
                if (o > bs) { bs = o; best = k; }
            }
        }
        if (lane == 0) {
            nu[i] = s > 0.f ? F / s : 0.f;
            kopt[i] = best;
        }
    }
}

// cell of a centroid: the frame [-1/2, W - 1/2) in cells of side cs, clamped
__device__ __forceinline__ int iso_cell(double x, double y, double cs, int ncx, int ncy)
{
    int cx = (int)floor((x + 0.5) / cs), cy = (int)floor((y + 0.5) / cs);
    cx = cx < 0 ? 0 : (cx >= ncx ? ncx - 1 : cx);
    cy = cy < 0 ? 0 : (cy >= ncy ? ncy - 1 : cy);
    return cy * ncx + cx;
}

__global__ void __launch_bounds__(256) k_iso_count(const double* __restrict__ xs, const double* __restrict__ ys,
                                                   const int* __restrict__ n_dev, int cap, double cs, int ncx, int ncy,
                                                   int* count)
{
    const int n = min(*n_dev, cap);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        atomicAdd(count + iso_cell(xs[i], ys[i], cs, ncx, ncy), 1);
}

// exclusive scan of count into start (one CTA, 8 cells a thread at a time);
// fill cleared
__global__ void __launch_bounds__(1024) k_iso_scan(const int* __restrict__ count, int ncell, int* start, int* fill)
{
    constexpr int V = 8;
    __shared__ int part[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int carry = 0;
    for (int c0 = 0; c0 < ncell; c0 += 1024 * V) {
        const int i0 = c0 + t * V;
        int v[V], sum = 0;
        const bool full = i0 + V <= ncell;       // 16-byte accesses (the arrays are 256-byte aligned)
        if (full) {
            const int4 a = reinterpret_cast<const int4*>(count + i0)[0], b = reinterpret_cast<const int4*>(count + i0)[1];
            v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
        } else {
#pragma unroll
            for (int k = 0; k < V; ++k) v[k] = i0 + k < ncell ? count[i0 + k] : 0;
        }
#pragma unroll
        for (int k = 0; k < V; ++k) sum += v[k];
        int inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        __syncthreads();                 // the last chunk's parts are read
        if (lane == 31) part[w] = inc;
        __syncthreads();
        int p = part[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, p, o);
            if (lane >= o) p += y;
        }
        const int before = __shfl_sync(0xffffffffu, p, w ? w - 1 : 0);
        int e = carry + (w ? before : 0) + inc - sum;
        int s[V];
#pragma unroll
        for (int k = 0; k < V; ++k) {
            s[k] = e;
            e += v[k];
        }
        if (full) {
            reinterpret_cast<int4*>(start + i0)[0] = make_int4(s[0], s[1], s[2], s[3]);
            reinterpret_cast<int4*>(start + i0)[1] = make_int4(s[4], s[5], s[6], s[7]);
            reinterpret_cast<int4*>(fill + i0)[0] = make_int4(0, 0, 0, 0);
            reinterpret_cast<int4*>(fill + i0)[1] = make_int4(0, 0, 0, 0);
        } else {
#pragma unroll
            for (int k = 0; k < V; ++k)
                if (i0 + k < ncell) {
                    start[i0 + k] = s[k];
                    fill[i0 + k] = 0;
                }
        }
        carry += __shfl_sync(0xffffffffu, p, 31);
    }
}

__global__ void __launch_bounds__(256) k_iso_fill(const double* __restrict__ xs, const double* __restrict__ ys,
                                                  const int* __restrict__ n_dev, int cap, double cs, int ncx, int ncy,
                                                  const int* __restrict__ start, int* fill, int* items)
{
    const int n = min(*n_dev, cap);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int c = iso_cell(xs[i], ys[i], cs, ncx, ncy);
        items[start[c] + atomicAdd(fill + c, 1)] = i;
    }
}

// Sums of the fit over some calibrators: their number, means of x = log10 nu
// and y = log10 r, the centred sums of squares and products, the range of x.
struct FitPart {
    double c, mx, my, sxx, sxy, lo, hi;
};
static_assert(sizeof(FitPart) == ROPT_PART_DOUBLES * sizeof(double), "the workspace holds a part of this size per CTA");

// two sets as one (the pairwise update of centred sums)
__device__ __forceinline__ FitPart fit_merge(const FitPart& a, const FitPart& b)
{
    if (a.c == 0.0) return b;
    if (b.c == 0.0) return a;
    FitPart r;
    r.c = a.c + b.c;
    const double dx = b.mx - a.mx, dy = b.my - a.my, f = b.c / r.c, g = a.c * f;
    r.mx = fma(dx, f, a.mx);
    r.my = fma(dy, f, a.my);
    r.sxx = fma(dx * dx, g, a.sxx + b.sxx);
    r.sxy = fma(dx * dy, g, a.sxy + b.sxy);
    r.lo = b.lo < a.lo ? b.lo : a.lo;
    r.hi = b.hi > a.hi ? b.hi : a.hi;
    return r;
}

// over the warp's lanes in a fixed tree, complete in lane 0
__device__ __forceinline__ FitPart fit_warp(FitPart v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        FitPart w;
        w.c = __shfl_down_sync(0xffffffffu, v.c, o); w.mx = __shfl_down_sync(0xffffffffu, v.mx, o);
        w.my = __shfl_down_sync(0xffffffffu, v.my, o); w.sxx = __shfl_down_sync(0xffffffffu, v.sxx, o);
        w.sxy = __shfl_down_sync(0xffffffffu, v.sxy, o); w.lo = __shfl_down_sync(0xffffffffu, v.lo, o);
        w.hi = __shfl_down_sync(0xffffffffu, v.hi, o);
        if (lane < o) v = fit_merge(v, w);
    }
    return v;
}

constexpr int CAL_NT = ROPT_PART_ROWS;

// The calibrator test (cheap conditions first, then the isolation: no other
// centroid closer than d_iso), and each CTA's part of the fit: float64 sums of
// every calibrator in one CTA are bound by its SM's float64 rate (56 us for
// 15,000 rows; 31 us for this test with 59 CTAs; 24 and 14 now).
__global__ void __launch_bounds__(CAL_NT) k_iso_calib(const double* __restrict__ xs, const double* __restrict__ ys,
                                                      const int* __restrict__ n_dev, int cap, double cs, int ncx, int ncy,
                                                      double d_iso, const int* __restrict__ start,
                                                      const int* __restrict__ count, const int* __restrict__ items,
                                                      const uint32_t* __restrict__ cflags,
                                                      const uint32_t* __restrict__ gflags, const double* __restrict__ flux,
                                                      const double* __restrict__ ferr, const float* __restrict__ nu,
                                                      const int* __restrict__ kopt, int nr, double snr_min,
                                                      const __grid_constant__ RoptRadii rad, uint8_t* calib, FitPart* parts)
{
    __shared__ FitPart part[CAL_NT / 32];
    const int n = min(*n_dev, cap);
    const double d2 = d_iso * d_iso;
    FitPart mine = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int ko = kopt[i];
        const double e = ferr[(int64_t)i * nr + ko];
        bool ok = cflags[i] == 0u && nu[i] > 0.f && (e > 0.0 ? flux[(int64_t)i * nr + ko] / e : 0.0) >= snr_min;
        uint32_t gf = 0u;
        if (ok)
            for (int k = 0; k < nr; ++k) gf |= gflags[(int64_t)i * nr + k];
        ok = ok && gf == 0u;
        if (ok) {
            const double x = xs[i], y = ys[i];
            const int c = iso_cell(x, y, cs, ncx, ncy), cx = c % ncx, cy = c / ncx;
            for (int gy = max(cy - 1, 0); gy <= min(cy + 1, ncy - 1) && ok; ++gy)
                for (int gx = max(cx - 1, 0); gx <= min(cx + 1, ncx - 1) && ok; ++gx) {
                    const int g = gy * ncx + gx;
                    for (int q = start[g]; q < start[g] + count[g]; ++q) {
                        const int j = items[q];
                        if (j == i) continue;
                        const double dx = xs[j] - x, dy = ys[j] - y;
                        if (dx * dx + dy * dy < d2) { ok = false; break; }
                    }
                }
        }
        calib[i] = ok ? 1 : 0;
        if (ok) {
            const double x = log10((double)nu[i]);
            mine = fit_merge(mine, FitPart{1.0, x, log10((double)rad.r[ko]), 0.0, 0.0, x, x});
        }
    }
    mine = fit_warp(mine);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < CAL_NT / 32; ++w) mine = fit_merge(mine, part[w]);
        parts[blockIdx.x] = mine;
    }
}

// the CTAs' parts (in a fixed order), then the line
constexpr int FIT_NT = 256;
__global__ void __launch_bounds__(FIT_NT) k_ropt_fit(const FitPart* __restrict__ parts, int nparts, double* fit)
{
    __shared__ FitPart part[FIT_NT / 32];
    FitPart v = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int i = threadIdx.x; i < nparts; i += FIT_NT) v = fit_merge(v, parts[i]);
    v = fit_warp(v);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    v = threadIdx.x < FIT_NT / 32 ? part[threadIdx.x] : FitPart{0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    v = fit_warp(v);
    if (threadIdx.x != 0) return;
    if (v.c < 3.0 || !(v.hi > v.lo)) {
        fit[0] = NAN; fit[1] = NAN; fit[2] = v.c; fit[3] = 1.0;
        return;
    }
    // a calibrator of radius 0 (log10 r = -inf) leaves no line, whichever
    // merge brought it in: some give an infinite slope where centred sums
    // about the common mean are NaN
    const double a = isfinite(v.mx) && isfinite(v.my) ? v.sxy / v.sxx : (double)NAN;
    fit[0] = a; fit[1] = v.my - a * v.mx; fit[2] = v.c; fit[3] = 0.0;
}

__global__ void __launch_bounds__(256) k_ropt_assign(const int* __restrict__ n_dev, int cap,
                                                     const uint8_t* __restrict__ calib, const float* __restrict__ nu,
                                                     const int* __restrict__ kopt,
                                                     const __grid_constant__ RoptRadii rad,
                                                     const double* __restrict__ fit, const double* __restrict__ flux,
                                                     const double* __restrict__ ferr, int* kfinal, double* flux_opt,
                                                     double* ferr_opt)
{
    const int n = min(*n_dev, cap);
    const int nr = rad.nr;
    const double a = fit[0], b = fit[1];
    const bool ok = fit[3] == 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        int k = 0;
        if (calib[i]) {
            k = kopt[i];
        } else if (ok && nu[i] > 0.f) {
            const double rf = exp10(fma(a, log10((double)nu[i]), b));
            double bd = INFINITY;
            for (int q = 0; q < nr; ++q) {
                const double d = fabs((double)rad.r[q] - rf);
                if (d <= bd) { bd = d; k = q; }      // ascending radii: ties go to the larger
            }
        }
        kfinal[i] = k;
        flux_opt[i] = flux[(int64_t)i * nr + k];
        ferr_opt[i] = ferr[(int64_t)i * nr + k];
    }
}

// cells of side cs >= d_iso, at most about 2^20 of them
void iso_grid(int W, int H, float d_iso, double* cs, int* ncx, int* ncy)
{
    double c = d_iso > 1.f ? (double)d_iso : 1.0;
    const double floor_c = ceil(sqrt((double)W * (double)H / (double)(1 << 20)));
    if (c < floor_c) c = floor_c;
    *cs = c;
    *ncx = (int)ceil((double)W / c) + 1;
    *ncy = (int)ceil((double)H / c) + 1;
}

cudaError_t launch_ropt(const Image& im, const SplineTab& sb, const SplineTab& sr, const float* taps, int kw, int kh,
                        const gp_catalog& cat, const double* flux, const double* ferr, const uint32_t* gflags,
                        const int* radii, int nr, float snr_min, float d_iso, const RoptWork& w, float* nu,
                        int* kopt, uint8_t* calib, int* kfinal, double* flux_opt, double* ferr_opt, double* fit,
                        cudaStream_t st)
{
    RoptRadii R;
    memset(&R, 0, sizeof R);
    R.nr = nr;
    for (int k = 0; k < nr; ++k) R.r[k] = radii[k];
    RoptTaps K;
    memset(&K, 0, sizeof K);
    K.kw = kw; K.kh = kh;
    for (int i = 0; i < kw * kh; ++i) K.t[i] = taps[i];
    const int cap = cat.capacity;
    const int grid = std::max(1, std::min((cap + 255) / 256, 152 * 8));
    const int rows = std::max(1, std::min((cap + 7) / 8, 152 * 32));     // 8 rows a CTA
    if (im.is_f32)
        k_ropt_nu<true><<<rows, 256, 0, st>>>(im, sb, sr, K, cat.xpeak, cat.ypeak, flux, ferr, nr, cat.n, cap, nu, kopt);
    else
        k_ropt_nu<false><<<rows, 256, 0, st>>>(im, sb, sr, K, cat.xpeak, cat.ypeak, flux, ferr, nr, cat.n, cap, nu,
                                               kopt);
    double cs;
    int ncx, ncy;
    iso_grid(im.W, im.H, d_iso, &cs, &ncx, &ncy);
    const int ncell = ncx * ncy;
    cudaError_t e = cudaMemsetAsync(w.count, 0, (size_t)ncell * sizeof(int), st);
    if (e != cudaSuccess) return e;
    k_iso_count<<<grid, 256, 0, st>>>(cat.x, cat.y, cat.n, cap, cs, ncx, ncy, w.count);
    k_iso_scan<<<1, 1024, 0, st>>>(w.count, ncell, w.start, w.fill);
    k_iso_fill<<<grid, 256, 0, st>>>(cat.x, cat.y, cat.n, cap, cs, ncx, ncy, w.start, w.fill, w.items);
    const int cal = ropt_parts(cap);
    FitPart* parts = reinterpret_cast<FitPart*>(w.parts);
    k_iso_calib<<<cal, CAL_NT, 0, st>>>(cat.x, cat.y, cat.n, cap, cs, ncx, ncy, (double)d_iso, w.start, w.count, w.items,
                                        cat.flags, gflags, flux, ferr, nu, kopt, nr, (double)snr_min, R, calib, parts);
    k_ropt_fit<<<1, FIT_NT, 0, st>>>(parts, cal, fit);
    k_ropt_assign<<<grid, 256, 0, st>>>(cat.n, cap, calib, nu, kopt, R, fit, flux, ferr, kfinal, flux_opt, ferr_opt);
    return cudaGetLastError();
}

}  // namespace gp
