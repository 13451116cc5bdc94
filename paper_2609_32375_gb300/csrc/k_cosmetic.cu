// k_cosmetic.cu -- the optional cosmetic corrections that precede the
// background (paper Section 3.1):
//
//  k_cr   the cosmic-ray filter, in the manner of L.A.Cosmic at the native
//         scale: L = 4 I - (the four nearest neighbours), L+ = max(L, 0);
//         the noise N = sqrt(max(med5(I), 0) gain + rn^2) / gain;
//         S = L+ / (sqrt(20) N) less its 5 x 5 median; the fine structure
//         F = med3(I) - med7(med3(I)), at least 0.01; a pixel is flagged when
//         S > sigclip and L+ / F > objlim, and takes the median of the good
//         unflagged pixels of its 5 x 5 window (unchanged if there are none).
//  k_rtn  the salt-and-pepper filter for random telegraph noise: a pixel whose
//         residual from its 3 x 3 median exceeds t in magnitude, with no such
//         pixel among its 8 neighbours, takes the median.
//
// Windows have a mirror border; bad pixels (masked or non-finite) are left
// out of every window (medians over the rest; the mean of the two middle
// values for an even count) and are never flagged or changed.
//
// Both filters change few pixels, so both first ask a cheap question whose
// "no" is certain, and take the medians only where the answer is "maybe":
//   k_rtn  the 3 x 3 median lies between the smallest and the largest of the
//          window's three row medians (small frames: every median, by blocks);
//   k_cr   med5(I) is at least the smallest of the window's five column
//          medians (15 of the 25 values are no less), which bounds S from
//          above before its own median is taken off (that is never negative).
// Windows without a bad pixel take the median-selection networks of
// median_sel.cuh, which find the same order statistic with about half the
// comparisons of a full sort.  A map value at a position outside the frame,
// computed from mirrored pixels, equals the mirrored map value, so the parts
// agree with whole-frame maps.
#include <math.h>

#include <type_traits>

#include "gp_internal.cuh"
#include "gp_launch.h"
#include "median_sel.cuh"

namespace gp {

constexpr int CM_B = 32;        // output block side
constexpr int CM_NT = 256;

// Batcher's odd-even merge sort of P (a power of two) values in registers,
// generated by compile-time recursion: sort both halves, then merge the
// elements R apart, the even and odd subsequences first; every comparator
// index is a template constant
__device__ __forceinline__ void cswap(float& a, float& b)
{
    const float lo = fminf(a, b), hi = fmaxf(a, b);
    a = lo;
    b = hi;
}

template <int LO, int N, int R, int P>
struct OEMerge {
    static __device__ __forceinline__ void run(float (&v)[P])
    {
        constexpr int step = R * 2;
        if constexpr (step < N) {
            OEMerge<LO, N, step, P>::run(v);
            OEMerge<LO + R, N, step, P>::run(v);
#pragma unroll
            for (int i = LO + R; i + R < LO + N; i += step) cswap(v[i], v[i + R]);
        } else {
            cswap(v[LO], v[LO + R]);
        }
    }
};

template <int LO, int N, int P>
struct OESort {
    static __device__ __forceinline__ void run(float (&v)[P])
    {
        if constexpr (N > 1) {
            OESort<LO, N / 2, P>::run(v);
            OESort<LO + N / 2, N / 2, P>::run(v);
            OEMerge<LO, N, 1, P>::run(v);
        }
    }
};

template <int P>
__device__ __forceinline__ void sort_net(float (&v)[P])
{
    OESort<0, P, P>::run(v);
}

// median of the non-NaN values among the N values in (N odd; NaN when none;
// the mean of the two middle values for an even count).  NaNs become +inf and
// -inf in turn, so that the middle values stand at fixed places: at places that
// follow from the count, the sorted values went through local memory.
template <int N, int P>
__device__ __forceinline__ float median_net(const float (&in)[N])
{
    static_assert(N % 2 == 1 && N < P, "an odd window, padded to a power of two");
    float v[P];
    unsigned bad = 0;
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const float x = i < N ? in[i] : INFINITY;
        const bool ok = !isnan(x);
        v[i] = ok ? x : __uint_as_float(0x7f800000u | bad << 31);
        bad += ok ? 0u : 1u;
    }
    sort_net<P>(v);
    const float a = v[N / 2], b = v[N / 2 - 1];
    return bad == N ? NAN : ((bad & 1u) ? 0.5f * (a + b) : a);
}

template <bool F32>
__device__ __forceinline__ float pixel_or_nan(const Image& im, int x, int y)
{
    bool bad;
    const float v = load_px<F32>(im, x, y, bad);
    return bad ? NAN : v;
}

// ------------------------------------------------------------------ CR ---
struct CrArgs {
    Image im;
    float gain, rn, sigclip, objlim;
    float* out;
    uint8_t* flags;          // nullable; bit 2 set where flagged
    int* count;              // nullable
};

// A CTA's 32 x 32 output pixels: flags for them and 2 pixels around (the fill
// windows), S 2 further (its median), pixels 2 further again (med5); med3 3
// around the flags, whose pixels lie 1 further.  Pixel columns are staged from
// X0 - 8, so that aligned frames stage 4 at a time.
constexpr int CR_F = CM_B + 4;           // flags, from (-2, -2)
constexpr int CR_S = CM_B + 8;           // S, from (-4, -4)
constexpr int CR_M = CM_B + 10;          // med3, from (-5, -5)
constexpr int CR_H = CM_B + 12;          // pixel rows, from -6
constexpr int CR_W = CM_B + 16;          // pixel columns, from -8

struct CrBlock {
    __align__(16) float a[CR_H][CR_W];
    __align__(16) float cm[CR_F][CR_S];  // vertical medians of 5 (rows from -2, columns from -4)
    uint8_t fl[CR_F][CR_F];
    uint16_t cand[CR_F * CR_F];
    int ncand, nflag;
};

// the whole maps, for blocks that hold a bad pixel
struct CrMaps {
    float S[CR_S][CR_S];
    float m3[CR_M][CR_M];
};

__device__ __forceinline__ float med5(float a, float b, float c, float d, float e)
{
    const float f = fmaxf(fminf(a, b), fminf(c, d)), g = fminf(fmaxf(a, b), fmaxf(c, d));
    return fmaxf(fminf(e, f), fminf(fmaxf(e, f), g));
}

__device__ __forceinline__ float cr_laplacian(const CrBlock& s, int r, int c)
{
    const float L = 4.f * s.a[r][c] - s.a[r][c - 1] - s.a[r][c + 1] - s.a[r - 1][c] - s.a[r + 1][c];
    return isnan(L) ? NAN : fmaxf(L, 0.f);
}

// S before its own median at pixel (r, c) of the stage
template <bool CLEAN>
__device__ __forceinline__ float cr_s(const CrBlock& s, const CrArgs& A, int r, int c)
{
    float v[25];
#pragma unroll
    for (int k = 0; k < 25; ++k) v[k] = s.a[r - 2 + k / 5][c - 2 + k % 5];
    float m5;
    if constexpr (CLEAN) m5 = med_sel<25>(v);
    else m5 = median_net<25, 32>(v);
    // NaN stays NaN here and below (fmaxf alone would return the other operand)
    const float noise = isnan(m5) ? NAN : sqrtf(fmaxf(m5, 0.f) * A.gain + A.rn * A.rn) / A.gain;
    return cr_laplacian(s, r, c) / (sqrtf(20.f) * noise);
}

template <bool CLEAN>
__device__ __forceinline__ float cr_m3(const CrBlock& s, int r, int c)
{
    float v[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = s.a[r - 1 + k / 3][c - 1 + k % 3];
    if constexpr (CLEAN) return med_sel<9>(v);
    else return median_net<9, 16>(v);
}

// every map at every position: blocks that hold a bad pixel, and ones with
// more candidates than this is worth skipping for
template <bool CLEAN>
__device__ __noinline__ void cr_flags_full(CrBlock& s, CrMaps& M, const CrArgs& A)
{
    const int t = threadIdx.x;
    for (int p = t; p < CR_M * CR_M; p += CM_NT) {
        const int r = p / CR_M, c = p - r * CR_M;
        M.m3[r][c] = cr_m3<CLEAN>(s, r + 1, c + 3);
    }
    for (int p = t; p < CR_S * CR_S; p += CM_NT) {
        const int r = p / CR_S, c = p - r * CR_S;
        M.S[r][c] = cr_s<CLEAN>(s, A, r + 2, c + 4);
    }
    __syncthreads();
    for (int p = t; p < CR_F * CR_F; p += CM_NT) {
        const int r = p / CR_F, c = p - r * CR_F;
        float v[25];
#pragma unroll
        for (int k = 0; k < 25; ++k) v[k] = M.S[r + k / 5][c + k % 5];
        float ms;
        if constexpr (CLEAN) ms = med_sel<25>(v);
        else ms = median_net<25, 32>(v);
        bool f = !isnan(s.a[r + 4][c + 6]) && M.S[r + 2][c + 2] - ms > A.sigclip;
        if (f) {            // the fine structure only where the first test holds (few pixels)
            float u[49];
#pragma unroll
            for (int k = 0; k < 49; ++k) u[k] = M.m3[r + k / 7][c + k % 7];
            float m7;
            if constexpr (CLEAN) m7 = med_sel<49>(u);
            else m7 = median_net<49, 64>(u);
            const float d = M.m3[r + 3][c + 3] - m7;
            const float F = isnan(d) ? NAN : fmaxf(d, 0.01f);
            f = cr_laplacian(s, r + 4, c + 6) / F > A.objlim;
        }
        s.fl[r][c] = f ? 1 : 0;
    }
}

// the middle of the N values the lanes hold (value lane in a, value 32 + lane
// in b; no NaN), by counting the smaller ones
template <int N>
__device__ __forceinline__ float warp_median(float a, float b)
{
    const int lane = threadIdx.x & 31;
    int ra = 0, rb = 0;
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const float v = __shfl_sync(0xffffffffu, j < 32 ? a : b, j & 31);
        ra += v < a || (v == a && j < lane);
        if (N > 32) rb += v < b || (v == b && j < lane + 32);
    }
    const unsigned ha = __ballot_sync(0xffffffffu, lane < N && ra == N / 2);
    const unsigned hb = N > 32 ? __ballot_sync(0xffffffffu, lane + 32 < N && rb == N / 2) : 0u;
    return ha ? __shfl_sync(0xffffffffu, a, __ffs(ha) - 1) : __shfl_sync(0xffffffffu, b, hb ? __ffs(hb) - 1 : 0);
}

// the exact decision at flag (r, c) of a block without bad pixels, by a warp:
// a lane computes one of the 25 values of S, then one or two of the 49 of med3
__device__ __forceinline__ bool cr_decide(const CrBlock& s, const CrArgs& A, int r, int c)
{
    const int lane = threadIdx.x & 31;
    const int l = lane < 25 ? lane : 24;
    const float S = cr_s<true>(s, A, r + 2 + l / 5, c + 4 + l % 5);
    const float S0 = __shfl_sync(0xffffffffu, S, 12);
    if (!(S0 > A.sigclip)) return false;
    const float ms = warp_median<25>(S, 0.f);
    if (!(S0 - ms > A.sigclip)) return false;
    const int h = lane + 32 < 49 ? lane + 32 : 48;
    const float u = cr_m3<true>(s, r + 1 + lane / 7, c + 3 + lane % 7), w = cr_m3<true>(s, r + 1 + h / 7, c + 3 + h % 7);
    const float d = __shfl_sync(0xffffffffu, u, 24) - warp_median<49>(u, w);
    return cr_laplacian(s, r + 4, c + 6) / fmaxf(d, 0.01f) > A.objlim;
}

// a block without one: candidates by the bound on S, then a warp for each.
// Bound by latency: the staging and the bound take some 600 warp instructions a
// block, but the eight warps meet at barriers, and between two of them one or two
// decide a candidate by 25- and 49-value rank counts, one shuffle after
// another, while the others wait.  A candidate is some 700 instructions, the
// full maps 19,000 a block; so more than CR_MOST candidates take those.
constexpr int CR_MOST = 28;

__device__ __forceinline__ void cr_flags_clean(CrBlock& s, CrMaps& M, const CrArgs& A)
{
    const int t = threadIdx.x;
    // vertical medians: a thread takes 6 rows of a column
    if (t < CR_S * (CR_F / 6)) {
        const int c = t % CR_S, r0 = t / CR_S * 6;
        float v[10];
#pragma unroll
        for (int k = 0; k < 10; ++k) v[k] = s.a[r0 + 2 + k][c + 4];
#pragma unroll
        for (int k = 0; k < 6; ++k) s.cm[r0 + k][c] = med5(v[k], v[k + 1], v[k + 2], v[k + 3], v[k + 4]);
    }
    for (int p = t; p < (int)sizeof(s.fl) / 4; p += CM_NT) reinterpret_cast<uint32_t*>(s.fl)[p] = 0u;
    __syncthreads();
    // S > sigclip needs L+ > sigclip sqrt(20) N; compared as squares, with
    // 1e-5 to spare for their rounding (and for a square below the normal
    // floats, no bound).  NaN and overflow count as "maybe".
    const float q = fmaxf(A.sigclip, 0.f) * sqrtf(20.f) / A.gain, K = q * q * (1.f - 1e-5f);
    const bool all = A.sigclip < 0.f;    // S = 0 passes too
    for (int p = t; p < CR_F * (CR_F / 4); p += CM_NT) {
        const int r = p / (CR_F / 4), c = 4 * (p - r * (CR_F / 4));
        const float4 lo = *reinterpret_cast<const float4*>(&s.cm[r][c]);
        const float4 hi = *reinterpret_cast<const float4*>(&s.cm[r][c + 4]);
        const float w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        // pixel (r, c) of the flags is pixel (r + 4, c + 6) of the stage
        const auto pair = [&](int dr, int dc) { return *reinterpret_cast<const float2*>(&s.a[r + 4 + dr][c + 6 + dc]); };
        const float2 x1 = pair(0, 0), x2 = pair(0, 2), u1 = pair(-1, 0), u2 = pair(-1, 2), d1 = pair(1, 0), d2 = pair(1, 2);
        const float x[6] = {s.a[r + 4][c + 5], x1.x, x1.y, x2.x, x2.y, s.a[r + 4][c + 10]};
        const float u[4] = {u1.x, u1.y, u2.x, u2.y}, d[4] = {d1.x, d1.y, d2.x, d2.y};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float m = fminf(fminf(fminf(w[e], w[e + 1]), fminf(w[e + 2], w[e + 3])), w[e + 4]);
            const float L = 4.f * x[e + 1] - x[e] - x[e + 2] - u[e] - d[e];
            const float l2 = L * L, n2 = K * fmaf(fmaxf(m, 0.f), A.gain, A.rn * A.rn);
            if ((all || !(L <= 0.f)) && (!(l2 < n2) || l2 < 1e-30f))
                s.cand[atomicAdd(&s.ncand, 1)] = (uint16_t)(r * CR_F + c + e);
        }
    }
    __syncthreads();
    const int ncand = s.ncand;
    if (ncand > CR_MOST) {
        cr_flags_full<true>(s, M, A);
        return;
    }
    for (int i = t >> 5; i < ncand; i += CM_NT / 32) {
        const int p = s.cand[i], r = p / CR_F, c = p - r * CR_F;
        if (cr_decide(s, A, r, c) && (t & 31) == 0) s.fl[r][c] = 1;
    }
}

// CLEAN: the frame cannot hold a bad pixel (uint16 without a mask); else
// each CTA looks whether its part does.  17 MP uint16: 804 us with every
// map computed at every pixel, 175 us so.  12 MP with one pixel in 500 masked, so
// that most blocks take the whole maps: 7.0 ms with the middle value picked from
// local memory, 0.86 so (median_net).
template <bool F32, bool CLEAN>
__global__ void __launch_bounds__(CM_NT, CLEAN ? 5 : 3) k_cr(const __grid_constant__ CrArgs A)
{
    __shared__ CrBlock s;
    __shared__ CrMaps maps;
    using T = typename std::conditional<F32, float, uint16_t>::type;
    const Image& im = A.im;
    const int W = im.W, H = im.H;
    const int X0 = blockIdx.x * CM_B, Y0 = blockIdx.y * CM_B;
    const int t = threadIdx.x;
    if (t == 0) s.ncand = s.nflag = 0;
    const T* data = reinterpret_cast<const T*>(im.data);
    const bool inside = X0 >= 8 && Y0 >= 6 && X0 - 8 + CR_W <= W && Y0 - 6 + CR_H <= H;
    bool odd = false;                    // a bad pixel, or a value whose sums could overflow
    if (inside && !im.mask && (im.pitch & 3) == 0 && (((uintptr_t)data) & (4 * sizeof(T) - 1)) == 0) {
        for (int p = t; p < CR_H * (CR_W / 4); p += CM_NT) {
            const int r = p / (CR_W / 4), c = 4 * (p - r * (CR_W / 4));
            const T* src = data + (int64_t)(Y0 - 6 + r) * im.pitch + X0 - 8 + c;
            float4 v;
            if constexpr (F32) {
                v = __ldg(reinterpret_cast<const float4*>(src));
                // bad pixels become NaN, as pixel_or_nan has them
                v.x = isfinite(v.x) ? v.x : NAN; v.y = isfinite(v.y) ? v.y : NAN;
                v.z = isfinite(v.z) ? v.z : NAN; v.w = isfinite(v.w) ? v.w : NAN;
                odd = odd || !(fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))) < 1e30f) ||
                      v.x != v.x || v.y != v.y || v.z != v.z || v.w != v.w;
            } else {
                const uint2 w = __ldg(reinterpret_cast<const uint2*>(src));
                v = make_float4((float)(w.x & 0xffffu), (float)(w.x >> 16), (float)(w.y & 0xffffu), (float)(w.y >> 16));
            }
            *reinterpret_cast<float4*>(&s.a[r][c]) = v;
        }
    } else {
        for (int p = t; p < CR_H * CR_W; p += CM_NT) {
            const int r = p / CR_W, c = p - r * CR_W;
            int x = X0 - 8 + c, y = Y0 - 6 + r;
            if ((unsigned)x >= (unsigned)W) x = mirror_idx(x, W);
            if ((unsigned)y >= (unsigned)H) y = mirror_idx(y, H);
            const float v = pixel_or_nan<F32>(im, x, y);
            s.a[r][c] = v;
            if (!CLEAN) odd = odd || !(fabsf(v) < 1e30f);
        }
    }
    if constexpr (CLEAN) {
        __syncthreads();
        cr_flags_clean(s, maps, A);
    } else {
        if (__syncthreads_or(odd)) cr_flags_full<false>(s, maps, A);
        else cr_flags_clean(s, maps, A);
    }
    __syncthreads();
    // 4 pixels of a row a thread
    static_assert(CM_NT * 4 == CM_B * CM_B, "one group of 4 a thread");
    const int r = t / (CM_B / 4), c0 = 4 * (t % (CM_B / 4));
    const int y = Y0 + r;
    if (y < H) {
        float o[4];
        uint32_t f4 = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int c = c0 + e;
            o[e] = s.a[r + 6][c + 8];
            if (!CLEAN && o[e] != o[e] && X0 + c < W) {      // a bad pixel keeps its value
                bool bad;
                o[e] = load_px<F32>(im, X0 + c, y, bad);
            }
            if (s.fl[r + 2][c + 2] && X0 + c < W) {
                float v[25];
#pragma unroll
                for (int k = 0; k < 25; ++k) {
                    const int dy = k / 5 - 2, dx = k % 5 - 2;
                    v[k] = s.fl[r + 2 + dy][c + 2 + dx] ? NAN : s.a[r + 6 + dy][c + 8 + dx];
                }
                const float m = median_net<25, 32>(v);
                o[e] = isnan(m) ? s.a[r + 6][c + 8] : m;
                f4 |= 2u << (8 * e);
                atomicAdd(&s.nflag, 1);
            }
        }
        const int64_t i = (int64_t)y * W + X0 + c0;
        if (X0 + c0 + 4 <= W && (W & 3) == 0 && (((uintptr_t)A.out) & 15) == 0) {
            *reinterpret_cast<float4*>(A.out + i) = make_float4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (X0 + c0 + e < W) A.out[i + e] = o[e];
        }
        if (A.flags) {
            if (X0 + c0 + 4 <= W && (W & 3) == 0 && (((uintptr_t)A.flags) & 3) == 0) {
                *reinterpret_cast<uint32_t*>(A.flags + i) = f4;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (X0 + c0 + e < W) A.flags[i + e] = (uint8_t)(f4 >> (8 * e));
            }
        }
    }
    __syncthreads();
    if (t == 0 && A.count && s.nflag) atomicAdd(A.count, s.nflag);
}

// ----------------------------------------------------------------- RTN ---
struct RtnArgs {
    Image im;
    float t;
    float* out;
    uint8_t* flags;          // nullable; bit 1 set where replaced (ORed into what is there when `keep`)
    int keep;
    int* count;
};

// min and max that hand on a NaN
__device__ __forceinline__ float min_nan(float a, float b)
{
    float d;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ float max_nan(float a, float b)
{
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

__device__ __forceinline__ float med3_nan(float a, float b, float c)
{
    return max_nan(min_nan(a, b), min_nan(max_nan(a, b), c));
}

// the median of a window with bad pixels (out of line: it stands in the middle
// of k_rtn's row loop, four times)
struct Window {
    float v[9];
};
__device__ __noinline__ float median_bad(Window w)
{
    return median_net<9, 16>(w.v);
}

// A warp takes 128 columns, a lane 4 of them, over ROWS rows, with the
// medians of 3 along three rows in registers; neighbours' columns come by
// shuffle.  The window's median lies between the smallest and the largest of
// its three row medians (6 of the 9 values are no less than the smallest), so
// only a pixel more than t from one of those, or with a bad pixel in its
// window (NaN), can be an outlier.  Those take the median of the 9 values in
// registers; an outlier's 8 neighbours are then tested by 8 lanes, or by its
// own lane where a row holds many (a track).  Bound by the row loop's latency.
// 17 MP after the cosmic-ray filter: 153 us with the median taken at every pixel
// of 32 x 32 blocks in shared memory, 75 us so.
constexpr int RTN_NT = 64;
// lanes with outliers in a row: up to this many, the warp's lanes test one's
// neighbours together, a round trip each; more (a track along the row) and each
// lane tests its own, eight round trips at most for all
constexpr int RTN_FEW = 6;

template <bool F32, int ROWS>
__global__ void __launch_bounds__(RTN_NT) k_rtn(const __grid_constant__ RtnArgs A, bool vec, bool ovec)
{
    using T = typename std::conditional<F32, float, uint16_t>::type;
    const Image& im = A.im;
    const int W = im.W, H = im.H;
    const int lane = threadIdx.x & 31, nx = (W + 127) / 128;
    const int wid = blockIdx.x * (RTN_NT / 32) + (threadIdx.x >> 5);
    const int y0 = wid / nx * ROWS, x0 = (wid % nx) * 128 + 4 * lane;
    if (y0 >= H) return;
    const int y1 = min(y0 + ROWS, H);
    // the lane's columns in the frame (mirrored beyond it), and the ones
    // beside the warp's that lanes 0 and 31 fetch
    int mx[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) mx[e] = x0 + e < W ? x0 + e : mirror_idx(x0 + e, W);
    const int ex = mirror_idx(lane ? x0 + 4 : x0 - 1, W);
    const bool full = vec && x0 + 4 <= W;
    struct Row {
        float v[4], e;
    };
    auto fetch = [&](int y) {
        Row r;
        const int gy = (unsigned)y < (unsigned)H ? y : mirror_idx(y, H);
        const T* row = reinterpret_cast<const T*>(im.data) + (int64_t)gy * im.pitch;
        if (full) {
            if constexpr (F32) {
                const float4 q = __ldg(reinterpret_cast<const float4*>(row + x0));
                r.v[0] = q.x; r.v[1] = q.y; r.v[2] = q.z; r.v[3] = q.w;
            } else {
                const uint2 q = __ldg(reinterpret_cast<const uint2*>(row + x0));
                r.v[0] = (float)(q.x & 0xffffu); r.v[1] = (float)(q.x >> 16);
                r.v[2] = (float)(q.y & 0xffffu); r.v[3] = (float)(q.y >> 16);
            }
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) r.v[e] = (float)__ldg(row + mx[e]);
        }
        r.e = lane == 0 || lane == 31 ? (float)__ldg(row + ex) : 0.f;
        return r;
    };
    // medians of 3 along the row, bad pixels as NaN
    struct Meds {
        float m[4], w[6];
    };
    auto meds = [&](const Row& r, int y) {
        float w[6] = {0.f, r.v[0], r.v[1], r.v[2], r.v[3], 0.f};
        float edge = r.e;
        if (F32) {
#pragma unroll
            for (int e = 0; e < 4; ++e) w[e + 1] = isfinite(w[e + 1]) ? w[e + 1] : NAN;
            edge = isfinite(edge) ? edge : NAN;
        }
        if (im.mask) {
            const int gy = (unsigned)y < (unsigned)H ? y : mirror_idx(y, H);
            const uint8_t* m = im.mask + (int64_t)gy * W;
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (__ldg(m + mx[e])) w[e + 1] = NAN;
            if ((lane == 0 || lane == 31) && __ldg(m + ex)) edge = NAN;
        }
        const float l = __shfl_up_sync(0xffffffffu, w[4], 1), g = __shfl_down_sync(0xffffffffu, w[1], 1);
        w[0] = lane == 0 ? edge : l;
        w[5] = lane == 31 ? edge : g;
        Meds h;
#pragma unroll
        for (int e = 0; e < 4; ++e) h.m[e] = med3_nan(w[e], w[e + 1], w[e + 2]);
#pragma unroll
        for (int e = 0; e < 6; ++e) h.w[e] = w[e];
        return h;
    };
    auto inside = [](int i, int n) { return (unsigned)i < (unsigned)n ? i : mirror_idx(i, n); };
    // pixel (px, py) of the frame: is it more than t from its window's median
    auto outlier = [&](int px, int py, float* med) {
        float v[9];
        bool bad = false;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            v[k] = pixel_or_nan<F32>(im, inside(px - 1 + k % 3, W), inside(py - 1 + k / 3, H));
            bad = bad || isnan(v[k]);
        }
        const float x = v[4];
        *med = bad ? median_net<9, 16>(v) : med_sel<9>(v);
        return !isnan(x) && fabsf(x - *med) > A.t;       // NaN comparisons are false
    };
    int nrep = 0;
    Row cur = fetch(y0), next = fetch(y0 + 1);
    Meds up = meds(fetch(y0 - 1), y0 - 1), mid = meds(cur, y0);
    for (int y = y0; y < y1; ++y) {
        const Row ahead = fetch(y + 2);
        const Meds down = meds(next, y + 1);
        float o[4];
        float med[4];
        uint32_t f4 = 0, hits = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            o[e] = cur.v[e];
            med[e] = 0.f;
            const float lo = min_nan(min_nan(up.m[e], mid.m[e]), down.m[e]);
            const float hi = max_nan(max_nan(up.m[e], mid.m[e]), down.m[e]);
            const bool maybe = !(max_nan(o[e] - lo, hi - o[e]) <= A.t) && x0 + e < W;
            if (!__any_sync(0xffffffffu, maybe)) continue;
            if (maybe) {
                Window w = {up.w[e], up.w[e + 1], up.w[e + 2], mid.w[e], mid.w[e + 1], mid.w[e + 2],
                            down.w[e], down.w[e + 1], down.w[e + 2]};
                const float x = mid.w[e + 1];                // NaN where the pixel is bad
                bool bad = false;
                if (F32 || im.mask) {
#pragma unroll
                    for (int k = 0; k < 9; ++k) bad = bad || isnan(w.v[k]);
                }
                med[e] = bad ? median_bad(w) : med_sel<9>(w.v);
                if (!isnan(x) && fabsf(x - med[e]) > A.t) hits |= 1u << e;      // NaN comparisons are false
            }
        }
        // an outlier is replaced when none of its neighbours is one
        unsigned b = __ballot_sync(0xffffffffu, hits != 0);
        if (__popc(b) <= RTN_FEW) {
            for (; b != 0; b = __ballot_sync(0xffffffffu, hits != 0)) {
                // one outlier, a neighbour a lane
                const int src = __ffs(b) - 1;
                const int e = __ffs(__shfl_sync(0xffffffffu, hits, src)) - 1;
                const int k = lane < 4 ? lane : lane + 1;
                const int px = __shfl_sync(0xffffffffu, x0, src) + e - 1 + k % 3, py = y - 1 + k / 3;
                float other;
                const bool hit = lane < 8 && outlier(inside(px, W), inside(py, H), &other);
                const bool alone = !__any_sync(0xffffffffu, hit);
                if (lane == src) {
                    hits &= hits - 1;
                    if (alone) f4 |= 1u << (8 * e);
                }
            }
        } else {
            // many: each lane its own
            for (; hits != 0; hits &= hits - 1) {
                const int e = __ffs(hits) - 1;
                bool alone = true;
                for (int k = 0; k < 9 && alone; ++k) {
                    float other;
                    if (k != 4 && outlier(inside(x0 + e - 1 + k % 3, W), inside(y - 1 + k / 3, H), &other))
                        alone = false;
                }
                if (alone) f4 |= 1u << (8 * e);
            }
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (f4 >> (8 * e) & 1u) {
                o[e] = med[e];
                ++nrep;
            }
        const int64_t i = (int64_t)y * W + x0;
        if (ovec && x0 + 4 <= W) {
            *reinterpret_cast<float4*>(A.out + i) = make_float4(o[0], o[1], o[2], o[3]);
            if (A.flags) {
                uint32_t* f = reinterpret_cast<uint32_t*>(A.flags + i);
                if (!A.keep) *f = f4;
                else if (f4) *f |= f4;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (x0 + e < W) {
                    A.out[i + e] = o[e];
                    const uint8_t f = (uint8_t)(f4 >> (8 * e));
                    if (A.flags && (!A.keep || f)) A.flags[i + e] = A.keep ? (uint8_t)(A.flags[i + e] | f) : f;
                }
        }
        up = mid;
        mid = down;
        cur = next;
        next = ahead;
    }
    nrep = __reduce_add_sync(0xffffffffu, nrep);
    if (lane == 0 && A.count && nrep) atomicAdd(A.count, nrep);
}

// Small frames: 32 x 32 blocks in shared memory, the median of every pixel.
// No step of it waits for a row's outliers, which set k_rtn's time where the
// chip is not filled.  CLEAN: the frame cannot hold a bad pixel (uint16 without a
// mask); else each CTA looks whether its part does.
template <bool F32, bool CLEAN>
__global__ void __launch_bounds__(CM_NT) k_rtn_block(const __grid_constant__ RtnArgs A)
{
    constexpr int HA = 2, NA = CM_B + 2 * HA;
    constexpr int HO = 1, NO = CM_B + 2 * HO;
    __shared__ float a[NA][NA];
    __shared__ float med[NO][NO];
    __shared__ uint8_t outl[NO][NO];
    __shared__ int nrep;
    const Image& im = A.im;
    const int W = im.W, H = im.H;
    const int X0 = blockIdx.x * CM_B, Y0 = blockIdx.y * CM_B;
    const int t = threadIdx.x;
    if (t == 0) nrep = 0;
    bool odd = false;
    for (int p = t; p < NA * NA; p += CM_NT) {
        const int r = p / NA, c = p - r * NA;
        const float v = pixel_or_nan<F32>(im, mirror_idx(X0 - HA + c, W), mirror_idx(Y0 - HA + r, H));
        a[r][c] = v;
        if (!CLEAN) odd = odd || isnan(v);
    }
    if constexpr (CLEAN) __syncthreads();
    else odd = __syncthreads_or(odd);
    for (int p = t; p < NO * NO; p += CM_NT) {
        const int r = p / NO, c = p - r * NO;
        float v[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) v[k] = a[r + k / 3][c + k % 3];
        float m;
        if (!CLEAN && odd) m = median_net<9, 16>(v);
        else m = med_sel<9>(v);
        const float x = a[r + 1][c + 1];
        med[r][c] = m;
        outl[r][c] = (!isnan(x) && fabsf(x - m) > A.t) ? 1 : 0;      // NaN comparisons are false
    }
    __syncthreads();
    for (int p = t; p < CM_B * CM_B; p += CM_NT) {
        const int r = p / CM_B, c = p - r * CM_B;
        const int x = X0 + c, y = Y0 + r;
        if (x >= W || y >= H) continue;
        bool rep = outl[r + 1][c + 1];
        for (int dy = 0; dy < 3 && rep; ++dy)
            for (int dx = 0; dx < 3; ++dx)
                if ((dy != 1 || dx != 1) && outl[r + dy][c + dx]) { rep = false; break; }
        bool unused;
        const int64_t i = (int64_t)y * W + x;
        A.out[i] = rep ? med[r + 1][c + 1] : load_px<F32>(im, x, y, unused);
        if (A.flags) {
            const uint8_t f = rep ? 1 : 0;
            A.flags[i] = A.keep ? (uint8_t)(A.flags[i] | f) : f;
        }
        if (rep) atomicAdd(&nrep, 1);
    }
    __syncthreads();
    if (t == 0 && A.count && nrep) atomicAdd(A.count, nrep);
}

cudaError_t launch_cr(const Image& im, float gain, float rn, float sigclip, float objlim, float* out, uint8_t* flags,
                      int* count, cudaStream_t st)
{
    CrArgs A;
    A.im = im; A.gain = gain; A.rn = rn; A.sigclip = sigclip; A.objlim = objlim;
    A.out = out; A.flags = flags; A.count = count;
    const dim3 g((im.W + CM_B - 1) / CM_B, (im.H + CM_B - 1) / CM_B);
    if (im.is_f32) k_cr<true, false><<<g, CM_NT, 0, st>>>(A);
    else if (im.mask) k_cr<false, false><<<g, CM_NT, 0, st>>>(A);
    else k_cr<false, true><<<g, CM_NT, 0, st>>>(A);
    return cudaGetLastError();
}

// Most pixels of a frame for the block form and for 2 rows a warp in place of 8
// (fewer rows read and sort more halo rows, but spread a small frame over more
// warps).  Blocks, 2 rows and 8 rows: 512 x 512 27, 45, 69 us; 1 MP 33, 36,
// 49; 2 MP 43, 46, 55; 4 MP 61, 51, 58; 12 MP 130, 109, 90; 17 MP 172, 138, 112
// (with windows that hold a bad pixel read again, which the last two no longer do).
constexpr int64_t RTN_BLOCK_PIXELS = 2 << 20, RTN_FEW_PIXELS = 6 << 20;

cudaError_t launch_rtn(const Image& im, float thr, float* out, uint8_t* flags, bool keep, int* count,
                       cudaStream_t st)
{
    RtnArgs A;
    A.im = im; A.t = thr; A.out = out; A.flags = flags; A.keep = keep ? 1 : 0; A.count = count;
    const int64_t pixels = (int64_t)im.W * im.H;
    if (pixels <= RTN_BLOCK_PIXELS && im.H <= 65535 * CM_B) {     // (a grid is 65,535 blocks high)
        const dim3 g((im.W + CM_B - 1) / CM_B, (im.H + CM_B - 1) / CM_B);
        if (im.is_f32) k_rtn_block<true, false><<<g, CM_NT, 0, st>>>(A);
        else if (im.mask) k_rtn_block<false, false><<<g, CM_NT, 0, st>>>(A);
        else k_rtn_block<false, true><<<g, CM_NT, 0, st>>>(A);
        return cudaGetLastError();
    }
    const bool vec = (im.pitch & 3) == 0 && (((uintptr_t)im.data) & (im.is_f32 ? 15 : 7)) == 0;
    const bool ovec = (im.W & 3) == 0 && (((uintptr_t)out) & 15) == 0 && (((uintptr_t)flags) & 3) == 0;
    auto run = [&](auto kern, int rows) {
        const int64_t warps = (int64_t)((im.W + 127) / 128) * ((im.H + rows - 1) / rows);
        kern<<<(int)((warps + RTN_NT / 32 - 1) / (RTN_NT / 32)), RTN_NT, 0, st>>>(A, vec, ovec);
    };
    if (pixels <= RTN_FEW_PIXELS) im.is_f32 ? run(k_rtn<true, 2>, 2) : run(k_rtn<false, 2>, 2);
    else im.is_f32 ? run(k_rtn<true, 8>, 8) : run(k_rtn<false, 8>, 8);
    return cudaGetLastError();
}

}  // namespace gp
