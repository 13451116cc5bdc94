// k_psf.cu -- the second detection pass with a spatially varying PSF (paper
// Section 3.2): the local PSF is a reference P0 plus K eigenmodes e_k with
// coefficient maps c_k, and the matched filter splits into K + 1
// correlations,
//     S(p) = (P0 (x) m)(p) + sum_k c_k(p) (e_k (x) m)(p),
// m = I - B (bad pixels 0, mirror border), c_k the natural spline through
// per-tile coefficients; foreground where S > k sigma(p).  The pass writes
// what the streaming threshold pass writes (packed mask, the map with m at
// foreground pixels and 0 elsewhere, the list of tiles holding foreground),
// so the labelling, merge and moments that follow are the plain path's.
//
// A CTA takes one 128-column strip and one 32-row tile band.  m over the band
// and a halo of KS/2 is formed in shared memory (four rows of a column at a
// time, which share the column's terms of the background spline); a thread
// takes one column and 16 rows and correlates them with two kernels at a
// time: per tap column it keeps the KS tap pairs in registers and walks the
// 16 + KS - 1 values of its column once, adding each to the rows that it
// reaches with paired FMAs (each half rounds as one fmaf, and each row meets its taps
// in order, so the results depend neither on the pairing nor on the walk).
// The taps (zero-padded to KS x KS, centred) are kernel parameters.
//
// Bound by the FMA pipe, two cycles a paired FMA: 13 x 13 taps, six kernels
// and 4096 x 4096 pixels are 266 M of them, 455 us.  It takes 630 us, and
// took 888 with 8 rows a thread (a third of its instructions were FMAs): the
// window's values copied into pairs half as often, and the splines' row
// terms from shared memory instead of divided out by every thread, are what
// went.
#include <math.h>
#include <string.h>

#include "gp_internal.cuh"
#include "gp_launch.h"

namespace gp {

constexpr int PS_ROWS = TY;                 // rows of a CTA: one tile band
constexpr int PS_COLS = ST_STRIP;           // columns: one mask strip (two tiles)
constexpr int PS_RPT = 16;                  // rows per thread
constexpr int PS_NT = PS_COLS * (PS_ROWS / PS_RPT);   // 256 threads
constexpr int PS_FILL = 4;                  // rows of a column filled together

// two FMAs with one rounding each, in one instruction (Blackwell's paired
// FP32 path): the lanes of a pair are independent, so the results are those
// of two fmaf
__device__ __forceinline__ float2 psf_ffma2(float2 a, float2 b, float2 c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;"
        : "=l"(d)
        : "l"(*reinterpret_cast<unsigned long long*>(&a)), "l"(*reinterpret_cast<unsigned long long*>(&b)),
          "l"(*reinterpret_cast<unsigned long long*>(&c)));
    return *reinterpret_cast<float2*>(&d);
}

constexpr int PS_NPAIR = (GP_PSF_MAX_MODES + 2) / 2;   // kernel pairs (P0 and the modes, a zero kernel last if odd)

struct PsfArgs {
    Image im;
    SplineTab sb, sr;
    SplineTab ct[GP_PSF_MAX_MODES];         // coefficient maps
    int nk;                                 // number of modes
    float thresh;
    uint32_t* seg;
    uint4* bits;
    int nstrip;
    int* tl_list;
    int* tl_count;
    Tiles T;
    float2 taps[PS_NPAIR][KMAX];             // kernels 2p and 2p + 1 of P0, then the modes: KS columns of KS taps
};

template <bool F32, int KS>
__global__ void __launch_bounds__(PS_NT, 3) k_psf(const __grid_constant__ PsfArgs A)
{
    constexpr int H = KS / 2, SR = PS_ROWS + KS - 1, SC = PS_COLS + KS - 1;
    __shared__ float ms[SR][SC];
    __shared__ float4 rowc[SR];            // b, c0, c1 of the background y-spline of each staged row
    __shared__ int2 rowj[SR];
    __shared__ float4 modec[GP_PSF_MAX_MODES][PS_ROWS];   // b, c0, c1, i of the modes' y-splines
    __shared__ uint8_t bads[PS_ROWS][PS_COLS];
    __shared__ uint32_t mbits[PS_ROWS][4];
    __shared__ int anyfg[2];
    const Image& im = A.im;
    const int W = im.W, Hf = im.H;
    const int X0 = blockIdx.x * PS_COLS, Y0 = blockIdx.y * PS_ROWS;
    const int t = threadIdx.x;
    for (int r = t; r < SR; r += PS_NT) {
        const AxCoef cy = axis_coef(A.sb.ay, (float)mirror_idx(Y0 - H + r, Hf));
        rowc[r] = make_float4(cy.b, cy.c0, cy.c1, 0.f);
        rowj[r] = make_int2(cy.i, cy.i1);
    }
    for (int q = t; q < A.nk * PS_ROWS; q += PS_NT) {
        const int k = q / PS_ROWS, r = q - k * PS_ROWS;
        const AxCoef cy = axis_coef(A.ct[k].ay, (float)min(Y0 + r, Hf - 1));
        modec[k][r] = make_float4(cy.b, cy.c0, cy.c1, __int_as_float(cy.i));
    }
    if (t < PS_ROWS * 4) mbits[t >> 2][t & 3] = 0u;
    if (t < 2) anyfg[t] = 0;
    __syncthreads();
    // ---- m over the band and its halo, PS_FILL rows of a column at a time
    // (consecutive threads take consecutive columns)
    constexpr int NF = (SR + PS_FILL - 1) / PS_FILL;
    for (int p = t; p < NF * SC; p += PS_NT) {
        const int g = p / SC, c = p - g * SC;
        const int x = mirror_idx(X0 - H + c, W);
        const AxCoef cx = axis_coef(A.sb.ax, (float)x);
        float val[PS_FILL];
        bool bad[PS_FILL];
#pragma unroll
        for (int j = 0; j < PS_FILL; ++j) {
            const int r = min(g * PS_FILL + j, SR - 1);
            val[j] = load_px<F32>(im, x, mirror_idx(Y0 - H + r, Hf), bad[j]);
        }
        int jc = -1;
        float2 b0 = make_float2(0.f, 0.f), b1 = b0;
#pragma unroll
        for (int j = 0; j < PS_FILL; ++j) {
            const int r = g * PS_FILL + j;
            if (r >= SR) break;
            const float4 rc = rowc[r];
            const int2 jy = rowj[r];
            if (jy.x != jc) {
                b0 = row_eval(A.sb, jy.x, cx);
                b1 = row_eval(A.sb, jy.y, cx);
                jc = jy.x;
            }
            AxCoef cy;
            cy.b = rc.x; cy.c0 = rc.y; cy.c1 = rc.z;
            ms[r][c] = bad[j] ? 0.f : val[j] - axis_combine(cy, b0.x, b1.x, b0.y, b1.y);
            const int ri = r - H, ci = c - H;
            if (ri >= 0 && ri < PS_ROWS && ci >= 0 && ci < PS_COLS) bads[ri][ci] = bad[j] ? 1 : 0;
        }
    }
    __syncthreads();
    // ---- the K + 1 correlations of this thread's column and rows
    const int col = t % PS_COLS, r0 = (t / PS_COLS) * PS_RPT;
    const int x = X0 + col;
    const bool xin = x < W;
    const int xq = xin ? x : W - 1;
    float S[PS_RPT];
#pragma unroll
    for (int r = 0; r < PS_RPT; ++r) S[r] = 0.f;
    const int npair = (A.nk + 2) / 2;
    for (int pr = 0; pr < npair; ++pr) {
        // kernels 2 pr and 2 pr + 1 together: one paired FMA per tap and row
        float2 F2[PS_RPT];
#pragma unroll
        for (int r = 0; r < PS_RPT; ++r) F2[r] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int u = 0; u < KS; ++u) {
            float2 tap[KS];
#pragma unroll
            for (int v = 0; v < KS; ++v) tap[v] = A.taps[pr][u * KS + v];
#pragma unroll
            for (int q = 0; q < PS_RPT + KS - 1; ++q) {
                const float a = ms[r0 + q][col + u];
                const float2 w = make_float2(a, a);
                // each row meets its taps v = 0, 1, .. in order
#pragma unroll
                for (int r = 0; r < PS_RPT; ++r)
                    if (q - r >= 0 && q - r < KS) F2[r] = psf_ffma2(tap[q - r], w, F2[r]);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = 2 * pr + h;
            if (k > A.nk) break;
            if (k == 0) {
#pragma unroll
                for (int r = 0; r < PS_RPT; ++r) S[r] = F2[r].x;
            } else {
                const SplineTab& ct = A.ct[k - 1];
                const AxCoef cx = axis_coef(ct.ax, (float)xq);
                int jc = -1;
                float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
                for (int r = 0; r < PS_RPT; ++r) {
                    const float4 rc = modec[k - 1][r0 + r];
                    const int j = __float_as_int(rc.w);
                    if (j != jc) {
                        a0 = row_eval(ct, j, cx);
                        a1 = row_eval(ct, min(j + 1, ct.ay.n - 1), cx);
                        jc = j;
                    }
                    AxCoef cy;
                    cy.b = rc.x; cy.c0 = rc.y; cy.c1 = rc.z;
                    S[r] = fmaf(axis_combine(cy, a0.x, a1.x, a0.y, a1.y), h ? F2[r].y : F2[r].x, S[r]);
                }
            }
        }
    }
    // ---- threshold, map, mask bits
    const AxCoef sx = axis_coef(A.sr.ax, (float)xq);
    uint32_t* srow = A.seg;
    int jc = -1;
    float2 q0 = make_float2(0.f, 0.f), q1 = q0;
#pragma unroll
    for (int r = 0; r < PS_RPT; ++r) {
        const int y = Y0 + r0 + r;
        if (!xin || y >= Hf) continue;
        // the noise map's axes are the background map's
        const float4 rc = rowc[r0 + r + H];
        const int2 jy = rowj[r0 + r + H];
        if (jy.x != jc) {
            q0 = row_eval(A.sr, jy.x, sx);
            q1 = row_eval(A.sr, jy.y, sx);
            jc = jy.x;
        }
        AxCoef sy;
        sy.b = rc.x; sy.c0 = rc.y; sy.c1 = rc.z;
        const float kt = A.thresh * axis_combine(sy, q0.x, q1.x, q0.y, q1.y);
        const bool fg = !bads[r0 + r][col] && S[r] > kt;
        const float mv = ms[r0 + r + H][col + H];
        srow[(int64_t)y * W + x] = fg ? __float_as_uint(mv) : 0u;
        if (fg) {
            atomicOr(&mbits[r0 + r][col & 3], 1u << (col >> 2));
            anyfg[col >> 6] = 1;
        }
    }
    __syncthreads();
    const int strip = blockIdx.x;
    if (t < PS_ROWS && Y0 + t < Hf)
        A.bits[(int64_t)(Y0 + t) * A.nstrip + strip] = make_uint4(mbits[t][0], mbits[t][1], mbits[t][2], mbits[t][3]);
    if (t < 2) {
        const int tcol = 2 * strip + t;
        if (tcol < A.T.ntx) {
            const int tile = blockIdx.y * A.T.ntx + tcol;
            if (anyfg[t]) A.tl_list[atomicAdd(A.tl_count, 1)] = tile;
            else A.T.piece_cnt[tile] = 0;
        }
    }
}

// the padded size of a kw x kh kernel (odd, at most 15)
static int psf_ks(int kw, int kh)
{
    const int k = kw > kh ? kw : kh;
    return k <= 3 ? 3 : k <= 5 ? 5 : k <= 7 ? 7 : k <= 9 ? 9 : k <= 11 ? 11 : k <= 13 ? 13 : 15;
}

template <int KS>
static cudaError_t launch_psf_ks(const PsfArgs& A, bool f32, dim3 g, cudaStream_t st)
{
    if (f32) k_psf<true, KS><<<g, PS_NT, 0, st>>>(A);
    else k_psf<false, KS><<<g, PS_NT, 0, st>>>(A);
    return cudaGetLastError();
}

cudaError_t launch_psf(const DetectArgs& D, const float* p0, const float* modes, int nk, int kw, int kh,
                       const SplineTab* coef_tabs, cudaStream_t st)
{
    PsfArgs A;
    memset(&A, 0, sizeof A);
    A.im = D.im; A.sb = D.sb; A.sr = D.sr;
    A.nk = nk;
    for (int k = 0; k < nk; ++k) A.ct[k] = coef_tabs[k];
    A.thresh = D.thresh;
    A.seg = D.seg; A.bits = D.bits; A.nstrip = D.nstrip;
    A.tl_list = D.tl_list; A.tl_count = D.tl_count; A.T = D.T;
    const int ks = psf_ks(kw, kh), ox = (ks - kw) / 2, oy = (ks - kh) / 2;
    for (int k = 0; k <= nk; ++k) {
        const float* src = k == 0 ? p0 : modes + (size_t)(k - 1) * kw * kh;
        for (int v = 0; v < kh; ++v)
            for (int u = 0; u < kw; ++u) {
                float2& t = A.taps[k / 2][(u + ox) * ks + (v + oy)];
                if (k & 1) t.y = src[v * kw + u];
                else t.x = src[v * kw + u];
            }
    }
    const dim3 g((D.im.W + PS_COLS - 1) / PS_COLS, (D.im.H + PS_ROWS - 1) / PS_ROWS);
    const bool f32 = D.im.is_f32;
    switch (ks) {
    case 3: return launch_psf_ks<3>(A, f32, g, st);
    case 5: return launch_psf_ks<5>(A, f32, g, st);
    case 7: return launch_psf_ks<7>(A, f32, g, st);
    case 9: return launch_psf_ks<9>(A, f32, g, st);
    case 11: return launch_psf_ks<11>(A, f32, g, st);
    case 13: return launch_psf_ks<13>(A, f32, g, st);
    default: return launch_psf_ks<15>(A, f32, g, st);
    }
}

}  // namespace gp
