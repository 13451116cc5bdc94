// k_cnn.cu -- the learned background: a small convolutional network that
// maps one-pass per-box quantile features (q10, q25, q50, q75, q90) to the
// background and rms meshes, replacing the iterative clip and median filter.
// The paper has no counterpart (its background is an FFT-smoothed local
// estimate, Section 3.1); the plain estimator stays as the fallback and as
// the source of the training targets.
//
// Network: six 3x3 convolutions (zero padding, same size) with ReLU between
// them, channels 5 -> 32 -> 48 -> 48 -> 32 -> 32 -> 2.  Activations are
// NHWC bfloat16 with channels padded to a multiple of 16; weights bfloat16,
// master weights and optimiser state float32; every contraction accumulates
// in float32.
//
//  k_conv3x3   implicit GEMM on the tensor cores (mma.sync m16n8k16 bf16):
//              one CTA per 64 output positions of four rows or of one, the
//              input patch and the whole weight matrix staged in shared memory.
//              Also computes the data gradient (with flipped, transposed
//              weights), gated by the layer's ReLU as it is stored.
//  k_wgrad     weight gradient dW[co][tap][ci] = sum_p dP[p][co] x[p+tap][ci]
//              as a tensor-core GEMM over positions, one partial per slot,
//              slots summed in a fixed order (reproducible).
//  k_update    AdamW of all layers and the packing of their weights.
//  others      ReLU backward, MSE loss, features, output denormalisation, and
//              packing and AdamW of one layer.
#include <cuda_bf16.h>
#include <math.h>

#include "block_select.cuh"
#include "gp_internal.cuh"
#include "gp_launch.h"

namespace gp {

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ void mma_bf16(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t ld_u32(const bf16* p) { return *reinterpret_cast<const uint32_t*>(p); }

__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi)
{
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__device__ __forceinline__ uint32_t smem_at(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// four 8 x 8 tiles of 16-bit values from shared memory into mma fragments;
// lane l names row l & 7 of tile l >> 3.  The transposed form hands out
// columns, so a tile stored [k][row] feeds an operand that wants [row][k].
__device__ __forceinline__ void ldm4(uint32_t* r, const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_at(p)) : "memory");
}

__device__ __forceinline__ void ldm4_trans(uint32_t* r, const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_at(p)) : "memory");
}

// 16 bytes global -> shared without a register stop; zeros when !ok
__device__ __forceinline__ void cp16(void* dst, const void* src, bool ok)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_at(dst)), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// a pair of bf16 gradients where the pair of activations y is positive (sign
// clear, not zero, not NaN), else 0
__device__ __forceinline__ uint32_t relu_gate(uint32_t y, uint32_t d)
{
    return (((y & 0xffffu) - 1u < 0x7f80u) ? d & 0xffffu : 0u) | (((y >> 16) - 1u < 0x7f80u) ? d & 0xffff0000u : 0u);
}

constexpr int CONV_TX = 64;      // output positions of a tile, along a row

// Rows of bf16 operands are staged 8 elements longer than they are: for 16,
// 32 and 48 channels (and 9 times as many weights) the 8 rows of an ldmatrix
// tile then start in 8 different 16-byte bank groups.
constexpr int SPAD = 8;

// ------------------------------------------------------------ forward ---
// Two tilings.  ROWS = 4 (8 warps of 32 positions: warp w takes half w & 1 of
// row w >> 1) reuses each weight fragment for two position tiles and stages
// six input rows for four output rows; its persistent CTAs keep the weights
// in shared memory from tile to tile.  ROWS = 1 (4 warps of 16 positions)
// spreads a single frame's few tiles over more SMs.  Either way an output
// accumulates its 9 x CIP products in the order tap, channel block, so both
// give the same bits.  Bound by the mma.sync rate: 48 to 48 channels at
// 131,072 positions take 21 us (257 TFLOP/s; 50 us when every 64 positions
// staged the weights anew and fragments came by 4-byte loads), a 64 x 64 mesh
// 5.5 us (10), most of it launch and staging latency.
template <int CIP, int COP, int ROWS>
struct ConvCfg {
    static constexpr int MT = ROWS == 1 ? 1 : 2;                     // 16-position tiles a warp
    static constexpr int NT = 32 * ROWS * CONV_TX / (16 * MT);       // threads
    static constexpr int PR = ROWS + 2, PC = CONV_TX + 2;            // patch rows and columns
    static constexpr int CS = CIP + SPAD, KS = 9 * CIP + SPAD;       // staged row lengths
    static constexpr size_t smem = sizeof(bf16) * ((size_t)PR * PC * CS + (size_t)COP * KS);
};

template <int CIP, int COP, int ROWS>
__global__ void __launch_bounds__(ConvCfg<CIP, COP, ROWS>::NT)
k_conv3x3(const bf16* __restrict__ x, const bf16* __restrict__ wt, const float* __restrict__ bias,
          void* __restrict__ y, int N, int H, int W, int relu, int out_f32, int creal, const bf16* __restrict__ gate)
{
    pdl_wait();
    pdl_release();
    using Cfg = ConvCfg<CIP, COP, ROWS>;
    constexpr int K = 9 * CIP, MT = Cfg::MT, NT = Cfg::NT, PR = Cfg::PR, PC = Cfg::PC, CS = Cfg::CS, KS = Cfg::KS;
    extern __shared__ __align__(16) unsigned char sm[];
    bf16* wts = reinterpret_cast<bf16*>(sm);                         // [COP][KS]
    bf16* patch = wts + COP * KS;                                    // [PR][PC][CS]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int q = tid; q < COP * K / 8; q += NT) {
        const int co = q / (K / 8), k = q - co * (K / 8);
        cp16(wts + co * KS + 8 * k, wt + (int64_t)q * 8, true);
    }
    const int g = lane >> 2, t = lane & 3;
    const int wrow = ROWS == 1 ? 0 : warp >> 1;                      // the warp's row and first position
    const int wx = ROWS == 1 ? warp * 16 : (warp & 1) * 32;
    // the lane's row of the ldmatrix tiles: positions (A), output channels (B)
    const int a_pos = ((lane >> 3) & 1) * 8 + (lane & 7), a_c = (lane >> 4) * 8;
    const int b_co = (lane >> 4) * 8 + (lane & 7), b_k = ((lane >> 3) & 1) * 8;
    const int nx = (W + CONV_TX - 1) / CONV_TX, ny = (H + ROWS - 1) / ROWS;
    const int64_t ntile = (int64_t)N * ny * nx;
    for (int64_t tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const int x0 = (int)(tile % nx) * CONV_TX;
        const int64_t ty = tile / nx;
        const int row0 = (int)(ty % ny) * ROWS, n = (int)(ty / ny);
        constexpr int VPP = CIP / 8;                                 // 16-byte vectors per position
        for (int q = tid; q < PR * PC * VPP; q += NT) {
            const int v = q % VPP, pc = q / VPP;
            const int r = pc / PC, c = pc - r * PC;
            const int gy = row0 + r - 1, gx = x0 + c - 1;
            const bool in = gy >= 0 && gy < H && gx >= 0 && gx < W;  // zero outside the mesh
            cp16(patch + pc * CS + v * 8, in ? x + (((int64_t)n * H + gy) * W + gx) * CIP + v * 8 : x, in);
        }
        cp_commit();
        cp_wait<0>();
        __syncthreads();
        float acc[MT][COP / 8][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < COP / 8; ++j) acc[m][j][0] = acc[m][j][1] = acc[m][j][2] = acc[m][j][3] = 0.f;
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
            const int dy = tap / 3, dx = tap % 3;
            const bf16* pa = patch + ((wrow + dy) * PC + wx + dx + a_pos) * CS + a_c;
#pragma unroll
            for (int cb = 0; cb < CIP / 16; ++cb) {
                uint32_t a[MT][4];
#pragma unroll
                for (int m = 0; m < MT; ++m) ldm4(a[m], pa + m * 16 * CS + cb * 16);
#pragma unroll
                for (int j = 0; j < COP / 8; j += 2) {
                    uint32_t b[4];
                    ldm4(b, wts + (j * 8 + b_co) * KS + tap * CIP + cb * 16 + b_k);
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        mma_bf16(acc[m][j], a[m][0], a[m][1], a[m][2], a[m][3], b[0], b[1]);
                        mma_bf16(acc[m][j + 1], a[m][0], a[m][1], a[m][2], a[m][3], b[2], b[3]);
                    }
                }
            }
        }
        // epilogue: bias, activation, store
        const int row = row0 + wrow;
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            const int gxa = x0 + wx + m * 16 + g, gxb = gxa + 8;
            if (row >= H) break;
#pragma unroll
            for (int j = 0; j < COP / 8; ++j) {
                const int co = j * 8 + 2 * t;
                const float* c = acc[m][j];
                const float b0 = bias ? bias[co] : 0.f, b1 = bias ? bias[co + 1] : 0.f;
                float v0 = c[0] + b0, v1 = c[1] + b1;
                float v2 = c[2] + b0, v3 = c[3] + b1;
                if (relu) { v0 = fmaxf(v0, 0.f); v1 = fmaxf(v1, 0.f); v2 = fmaxf(v2, 0.f); v3 = fmaxf(v3, 0.f); }
                if (out_f32) {
                    float* yo = reinterpret_cast<float*>(y);
                    if (gxa < W) {
                        const int64_t o = (((int64_t)n * H + row) * W + gxa) * creal;
                        if (co < creal) yo[o + co] = v0;
                        if (co + 1 < creal) yo[o + co + 1] = v1;
                    }
                    if (gxb < W) {
                        const int64_t o = (((int64_t)n * H + row) * W + gxb) * creal;
                        if (co < creal) yo[o + co] = v2;
                        if (co + 1 < creal) yo[o + co + 1] = v3;
                    }
                } else {
                    bf16* yo = reinterpret_cast<bf16*>(y);
                    const int64_t oa = (((int64_t)n * H + row) * W + gxa) * COP + co, ob = oa + 8 * COP;
                    const uint32_t pa = pack2(__float2bfloat16_rn(v0), __float2bfloat16_rn(v1));
                    const uint32_t pb = pack2(__float2bfloat16_rn(v2), __float2bfloat16_rn(v3));
                    if (gxa < W) *reinterpret_cast<uint32_t*>(yo + oa) = gate ? relu_gate(ld_u32(gate + oa), pa) : pa;
                    if (gxb < W) *reinterpret_cast<uint32_t*>(yo + ob) = gate ? relu_gate(ld_u32(gate + ob), pb) : pb;
                }
            }
        }
        __syncthreads();                                             // the patch is free again
    }
}

// ---------------------------------------------------- weight gradient ---
// Block (slot, dy): output rows r = slot, slot + nslot, ... of the N*H; a warp
// for each of the three taps (dy, dx) and each 16 output channels.  Bound by
// the mma.sync rate (about 5 cycles an SM for each m16n8k16, as in k_conv3x3)
// of the fullest SM: the caller chooses nslot, and with 152 (three blocks on
// every SM) the six layers and their reductions take 156 us, with 128 178, and with 64
// (two blocks on 40 SMs, one on the others) 235.
// 131,072 positions, 48 to 48 channels, 64 slots: 48 us; one warp a tap 53, element-wise
// transposed staging with a block a tap, which this replaced, 270.
// GEMM per 64 positions of a row: M = COP
// output channels, N = CIP input channels, K = positions.  dP and the input
// row are staged as they lie, by 16-byte asynchronous copies three chunks ahead,
// and the transposing ldmatrix gives both operands their [channel][position]
// fragments.  The blocks of dy = 1 also sum dP into the slot's bias gradient.
constexpr int WG_STAGES = 4;     // row chunks in flight: a chunk's products take less time than an L2 round trip
template <int CIP, int COP>
constexpr size_t wgrad_smem()
{
    return sizeof(bf16) * WG_STAGES * (size_t)(CONV_TX * (COP + SPAD) + (CONV_TX + 2) * (CIP + SPAD));
}

template <int CIP, int COP>
__global__ void __launch_bounds__(6 * COP) k_wgrad(const bf16* __restrict__ x, const bf16* __restrict__ dp, int NH,
                                                 int H, int W, int nslot, bool vec, float* __restrict__ partial,
                                                 float* __restrict__ bpart)
{
    pdl_wait();
    pdl_release();
    constexpr int DS = COP + SPAD, XS = CIP + SPAD;
    constexpr int NW = 3 * (COP / 16), WG_NT = 32 * NW;
    extern __shared__ __align__(16) unsigned char sm[];
    bf16 (*dps)[CONV_TX][DS] = reinterpret_cast<bf16 (*)[CONV_TX][DS]>(sm);    // dP: [stage][position][co]
    bf16 (*xs)[CONV_TX + 2][XS] = reinterpret_cast<bf16 (*)[CONV_TX + 2][XS]>(sm + sizeof(bf16) * WG_STAGES * CONV_TX * DS);
    __shared__ float bred[WG_NT][2];                                 // xs: input row, positions -1 .. 64
    const int tid = threadIdx.x, lane = tid & 31, dx = (tid >> 5) % 3, mt = (tid >> 5) / 3;
    const int slot = blockIdx.x, dy = blockIdx.y;
    const int g = lane >> 2, t = lane & 3;
    constexpr int NT = CIP / 8;
    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    // bias: thread = channel pair (tid % (COP / 2)), every BQ-th position
    constexpr int BP = COP / 2, BQ = WG_NT / BP;
    const int bc = tid % BP, bq = tid / BP;
    float b0 = 0.f, b1 = 0.f;
    const int nx = (W + CONV_TX - 1) / CONV_TX;
    const int nrow = slot < NH ? (NH - slot + nslot - 1) / nslot : 0, nchunk = nrow * nx;
    // 8 channels of one position (vec: both arrays are 16-byte aligned)
    auto put = [&](bf16* dst, const bf16* src, bool in) {
        if (vec) {
            cp16(dst, src, in);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) dst[e] = in ? src[e] : __float2bfloat16_rn(0.f);
        }
    };
    auto stage = [&](int c, int buf) {
        const int r = slot + (c / nx) * nslot, x0 = (c % nx) * CONV_TX;
        const int n = r / H, row = r - n * H, srow = row + dy - 1;
        const bool rin = srow >= 0 && srow < H;
        for (int q = tid; q < CONV_TX * (COP / 8); q += WG_NT) {
            const int p = q / (COP / 8), v = q - p * (COP / 8);
            const bool in = x0 + p < W;
            put(&dps[buf][p][8 * v], in ? dp + ((int64_t)r * W + x0 + p) * COP + 8 * v : dp, in);
        }
        for (int q = tid; q < (CONV_TX + 2) * (CIP / 8); q += WG_NT) {
            const int p = q / (CIP / 8), v = q - p * (CIP / 8), gx = x0 + p - 1;
            const bool in = rin && gx >= 0 && gx < W;
            put(&xs[buf][p][8 * v], in ? x + (((int64_t)n * H + srow) * W + gx) * CIP + 8 * v : x, in);
        }
    };
    for (int c = 0; c < WG_STAGES - 1; ++c) {
        if (c < nchunk) stage(c, c);
        cp_commit();
    }
    const int l8 = lane & 7, mi = lane >> 3;
    for (int c = 0; c < nchunk; ++c) {
        const int buf = c % WG_STAGES;
        cp_wait<WG_STAGES - 2>();
        __syncthreads();                                             // chunk c is in; chunk c - 1's stage is free
        if (c + WG_STAGES - 1 < nchunk) stage(c + WG_STAGES - 1, (c + WG_STAGES - 1) % WG_STAGES);
        cp_commit();
#pragma unroll
        for (int ks = 0; ks < CONV_TX / 16; ++ks) {
            uint32_t a[4];
            ldm4_trans(a, &dps[buf][ks * 16 + (mi >> 1) * 8 + l8][mt * 16 + (mi & 1) * 8]);
#pragma unroll
            for (int j = 0; j < NT; j += 2) {
                uint32_t b[4];
                ldm4_trans(b, &xs[buf][ks * 16 + (mi & 1) * 8 + l8 + dx][j * 8 + (mi >> 1) * 8]);
                mma_bf16(acc[j], a[0], a[1], a[2], a[3], b[0], b[1]);
                mma_bf16(acc[j + 1], a[0], a[1], a[2], a[3], b[2], b[3]);
            }
        }
        if (dy == 1 && bq < BQ) {
#pragma unroll 4
            for (int p = bq; p < CONV_TX; p += BQ) {
                const uint32_t w = ld_u32(&dps[buf][p][2 * bc]);
                b0 += __uint_as_float(w << 16);
                b1 += __uint_as_float(w & 0xffff0000u);
            }
        }
    }
    // partial[slot][tap][co][ci]
    float* out = partial + ((int64_t)slot * 9 + dy * 3 + dx) * COP * CIP;
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int co = mt * 16 + g, ci = j * 8 + 2 * t;
        out[co * CIP + ci] = acc[j][0];
        out[co * CIP + ci + 1] = acc[j][1];
        out[(co + 8) * CIP + ci] = acc[j][2];
        out[(co + 8) * CIP + ci + 1] = acc[j][3];
    }
    if (dy != 1) return;
    bred[tid][0] = b0;
    bred[tid][1] = b1;
    __syncthreads();
    if (tid < COP) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < BQ; ++q) s += bred[q * BP + (tid >> 1)][tid & 1];
        bpart[slot * COP + tid] = s;
    }
}

// dW[co][ci][3][3] (real channels) = sum over the slots in a fixed order, in
// the partials' own layout (the writes scatter); the last blocks sum the bias,
// whose partials k_wgrad makes from the dP it has staged (a kernel of its own
// with one position a step took 287 us of a layer's step, this 5).
// A warp takes every WR_PARTS-th slot of 32 outputs (the partials are read in
// 128-byte rows), and the warps' sums are added in order.
constexpr int WR_PARTS = 8;
__global__ void __launch_bounds__(32 * WR_PARTS)
k_wgrad_reduce(const float* __restrict__ partial, const float* __restrict__ bpart, int nslot, int cip, int cop, int cir,
               int cor, float* __restrict__ dw, float* __restrict__ db)
{
    pdl_wait();
    pdl_release();
    __shared__ float part[WR_PARTS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = 9 * cop * cip, nb = (per + 31) / 32;
    const bool isb = (int)blockIdx.x >= nb;                          // the bias gradients follow the weights'
    const int i = ((int)blockIdx.x - (isb ? nb : 0)) * 32 + lane, n = isb ? cop : per;
    const float* src = isb ? bpart : partial;
    float s = 0.f;
    if (i < n) {
#pragma unroll 8
        for (int k = warp; k < nslot; k += WR_PARTS) s += src[(int64_t)k * n + i];
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp || i >= n) return;
    s = part[0][lane];
#pragma unroll
    for (int p = 1; p < WR_PARTS; ++p) s += part[p][lane];
    if (isb) {
        if (i < cor) db[i] = s;
        return;
    }
    const int tap = i / (cop * cip), rem = i - tap * cop * cip, co = rem / cip, ci = rem - co * cip;
    if (co < cor && ci < cir) dw[(co * cir + ci) * 9 + tap] = s;
}

// -------------------------------------------------------- elementwise ---
// 8 values a thread where the three arrays are 16-byte aligned (nvec of
// them), the rest one by one
__global__ void k_relu_backward(const bf16* __restrict__ dy, const bf16* __restrict__ y, bf16* __restrict__ dp,
                                int64_t nvec, int64_t count)
{
    pdl_wait();
    pdl_release();
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < nvec; i += step) {
        const uint4 a = reinterpret_cast<const uint4*>(dy)[i], b = reinterpret_cast<const uint4*>(y)[i];
        const uint32_t av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = relu_gate(bv[e], av[e]);
        reinterpret_cast<uint4*>(dp)[i] = make_uint4(o[0], o[1], o[2], o[3]);
    }
    for (int64_t i = 8 * nvec + i0; i < count; i += step)
        dp[i] = __bfloat162float(y[i]) > 0.f ? dy[i] : __float2bfloat16_rn(0.f);
}

// mean squared error over npos positions x 2 channels; dY (bf16, padded to
// cop channels) = 2 (pred - target) / (2 npos); per-block partial losses
__global__ void k_mse(const float* __restrict__ pred, const float* __restrict__ target, int64_t npos, int cop,
                      bf16* __restrict__ dy, float* __restrict__ part)
{
    pdl_wait();
    pdl_release();
    __shared__ float red[256];
    float s = 0.f;
    const float scale = 2.f / (2.f * (float)npos);
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < npos; p += (int64_t)gridDim.x * blockDim.x) {
        for (int c = 0; c < cop; ++c) {
            float d = 0.f;
            if (c < 2) {
                d = pred[p * 2 + c] - target[p * 2 + c];
                s += d * d;
            }
            dy[p * cop + c] = __float2bfloat16_rn(scale * d);
        }
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// one warp, a fixed order
__global__ void k_mse_reduce(const float* __restrict__ part, int nb, int64_t npos, float* __restrict__ loss)
{
    pdl_wait();
    pdl_release();
    double s = 0.0;
    for (int i = threadIdx.x; i < nb; i += 32) s += part[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *loss = (float)(s / (2.0 * (double)npos));
}

// master W[co][ci][3][3] (real channels) -> forward wt[cop][9*cip] and the
// data-gradient weights wtd[cip][9*cop] (taps flipped, in and out swapped)
__global__ void k_pack(const float* __restrict__ W, const float* __restrict__ b, int cir, int cor, int cip, int cop,
                       bf16* __restrict__ wt, bf16* __restrict__ wtd, float* __restrict__ bias_p)
{
    pdl_wait();
    pdl_release();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < cop * 9 * cip) {
        const int co = i / (9 * cip), k = i - co * 9 * cip, tap = k / cip, ci = k - tap * cip;
        const float v = (co < cor && ci < cir) ? W[(co * cir + ci) * 9 + tap] : 0.f;
        wt[i] = __float2bfloat16_rn(v);
        // wtd[ci][tap' * cop + co] with tap' the flipped tap
        const int tf = 8 - tap;
        wtd[(int64_t)ci * 9 * cop + tf * cop + co] = __float2bfloat16_rn(v);
    }
    if (i < cop) bias_p[i] = i < cor ? b[i] : 0.f;
}

struct AdamW {
    float lr, b1, b2, eps, c1, c2;       // c1, c2: the bias corrections 1 - beta^step
};

// one value's step
__device__ __forceinline__ float adamw_step(const AdamW& o, float wd, float p, float g, float& m, float& v)
{
    m = o.b1 * m + (1.f - o.b1) * g;
    v = o.b2 * v + (1.f - o.b2) * g * g;
    const float mh = m / o.c1, vh = v / o.c2;
    return p - o.lr * (mh / (sqrtf(vh) + o.eps) + wd * p);
}

__global__ void k_adamw(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                        float* __restrict__ v, int64_t n, const __grid_constant__ AdamW o, float wd)
{
    pdl_wait();
    pdl_release();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float mi = m[i], vi = v[i];
        p[i] = adamw_step(o, wd, p[i], g[i], mi, vi);
        m[i] = mi;
        v[i] = vi;
    }
}

// AdamW of every layer's weights and biases and their packed forms, in one
// launch: layer blockIdx.y, a thread a weight, the biases in the last block.
// (Zeros beside the layer's own channels stay as k_pack left them.)  A step of the
// six-layer network: 4 us, 62 as twelve k_adamw and six k_pack.
__global__ void k_update(const __grid_constant__ CnnLayers L, const __grid_constant__ AdamW o, float wd)
{
    pdl_wait();
    pdl_release();
    const gp_cnn_layer& A = L.l[blockIdx.y];
    const int cir = A.cin, cor = A.cout, n = cor * cir * 9;
    if (blockIdx.x == gridDim.x - 1) {
        for (int i = threadIdx.x; i < cor; i += blockDim.x) {
            float mi = A.mb[i], vi = A.vb[i];
            const float p = adamw_step(o, 0.f, A.b[i], A.db[i], mi, vi);
            A.mb[i] = mi; A.vb[i] = vi; A.b[i] = p;
            A.bias_p[i] = p;
        }
        return;
    }
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float mi = A.mW[i], vi = A.vW[i];
    const float p = adamw_step(o, wd, A.W[i], A.dW[i], mi, vi);
    A.mW[i] = mi; A.vW[i] = vi; A.W[i] = p;
    const int tap = i % 9, cc = i / 9, co = cc / cir, ci = cc - co * cir;
    const bf16 q = __float2bfloat16_rn(p);
    reinterpret_cast<bf16*>(A.wt)[(int64_t)co * 9 * A.cin_p + tap * A.cin_p + ci] = q;
    reinterpret_cast<bf16*>(A.wtd)[(int64_t)ci * 9 * A.cout_p + (8 - tap) * A.cout_p + co] = q;
}

// ------------------------------------------------------------ features ---
// One CTA per frame: centre c = median of the box medians q50, scale
// s = median of (q75 - q25) / 1.349 (the Gaussian sigma of an interquartile
// range); features (q_k - c) / s in channels 0..4 of a 16-channel NHWC
// bf16 map; (c, s) kept for denormalising the output.  Bound by the latency
// of one CTA's passes: 18 us for 4,096 boxes (79 with two bitonic sorts and
// the features written one by one).
constexpr int FEAT_NT = 1024;

// median of the n values value(0) .. value(n - 1)
template <class Value>
__device__ float block_median(Value value, int n, SelShared<FEAT_NT>& S)
{
    auto each = [&](auto f) {
        for (int i = threadIdx.x; i < n; i += FEAT_NT) f(key_of(value(i)));
    };
    // the values' range first, so that block_select's bins cover no more
    uint32_t lo = 0xffffffffu, hi = 0u;
    each([&](uint32_t k) { lo = min(lo, k); hi = max(hi, k); });
    if (threadIdx.x == 0) { S.excl = 0xffffffffu; S.next = 0u; }
    __syncthreads();
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) { atomicMin(&S.excl, lo); atomicMax(&S.next, hi); }
    __syncthreads();
    lo = S.excl;
    hi = S.next;
    __syncthreads();
    uint32_t k1 = 0;
    const uint32_t k0 = block_select<FEAT_NT>(each, lo, hi, (uint32_t)(n - 1) / 2, (n & 1) ? nullptr : &k1, S);
    return (n & 1) ? key_value(k0) : 0.5f * (key_value(k0) + key_value(k1));
}

__global__ void __launch_bounds__(FEAT_NT) k_features(const float* __restrict__ quant, int nbox,
                                                      bf16* __restrict__ feat, float* __restrict__ norm)
{
    pdl_wait();
    pdl_release();
    __shared__ __align__(16) SelShared<FEAT_NT> sel;
    const int f = blockIdx.x;
    const float* q = quant + (int64_t)f * 5 * nbox;                  // [5][nbox]
    const float c = block_median([&](int i) { return __ldg(q + 2 * nbox + i); }, nbox, sel);
    __syncthreads();
    float s = block_median([&](int i) { return __ldg(q + 3 * nbox + i) - __ldg(q + nbox + i); }, nbox, sel) / 1.349f;
    if (!(s > 0.f)) s = 1.f;
    if (threadIdx.x == 0) { norm[2 * f] = c; norm[2 * f + 1] = s; }
    bf16* fo = feat + (int64_t)f * nbox * 16;
    const bool vec = (((uintptr_t)feat) & 15) == 0;
    for (int b = threadIdx.x; b < nbox; b += FEAT_NT) {
        bf16 v[16];
#pragma unroll
        for (int ch = 0; ch < 16; ++ch)
            v[ch] = __float2bfloat16_rn(ch < 5 ? (__ldg(q + ch * nbox + b) - c) / s : 0.f);
        if (vec) {
            uint4* o = reinterpret_cast<uint4*>(fo + (int64_t)b * 16);
            o[0] = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
            o[1] = make_uint4(0u, 0u, 0u, 0u);
        } else {
            for (int ch = 0; ch < 16; ++ch) fo[(int64_t)b * 16 + ch] = v[ch];
        }
    }
}

// network output (N x nbox x 2, normalised) -> meshes
__global__ void k_denorm(const float* __restrict__ out, const float* __restrict__ norm, int nbox, int64_t total,
                         float* __restrict__ bkg, float* __restrict__ rms)
{
    pdl_wait();
    pdl_release();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int f = (int)(i / nbox);
        const float c = norm[2 * f], s = norm[2 * f + 1];
        bkg[i] = c + s * out[2 * i];
        rms[i] = s * fmaxf(out[2 * i + 1], 0.f);
    }
}

// meshes -> normalised targets (training)
__global__ void k_targets(const float* __restrict__ bkg, const float* __restrict__ rms, const float* __restrict__ norm,
                          int nbox, int64_t total, float* __restrict__ tgt)
{
    pdl_wait();
    pdl_release();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int f = (int)(i / nbox);
        const float c = norm[2 * f], s = norm[2 * f + 1];
        tgt[2 * i] = (bkg[i] - c) / s;
        tgt[2 * i + 1] = rms[i] / s;
    }
}

// --------------------------------------------------------------- launchers ---
template <int CIP, int COP, int ROWS>
static cudaError_t conv_launch_rows(const void* x, int n, int h, int w, const void* wt, const float* bias, int relu,
                                    void* y, int out_f32, int creal, const void* gate, int64_t most, cudaStream_t st)
{
    using Cfg = ConvCfg<CIP, COP, ROWS>;
    cudaFuncSetAttribute(k_conv3x3<CIP, COP, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::smem);
    const int64_t ntile = (int64_t)n * ((h + ROWS - 1) / ROWS) * ((w + CONV_TX - 1) / CONV_TX);
    launch_dep(k_conv3x3<CIP, COP, ROWS>, dim3((int)(ntile < most ? ntile : most)), dim3(Cfg::NT), Cfg::smem, st,
               reinterpret_cast<const bf16*>(x), reinterpret_cast<const bf16*>(wt), bias, y, n, h, w, relu, out_f32,
               creal, reinterpret_cast<const bf16*>(gate));
    return cudaGetLastError();
}

template <int CIP, int COP>
static cudaError_t conv_launch(const void* x, int n, int h, int w, const void* wt, const float* bias, int relu,
                               void* y, int out_f32, int creal, const void* gate, cudaStream_t st)
{
    if (n <= 0 || h <= 0 || w <= 0) return cudaErrorInvalidConfiguration;
    // four-row tiles once there is one for every SM; below, single rows
    const int64_t tiles4 = (int64_t)n * ((h + 3) / 4) * ((w + CONV_TX - 1) / CONV_TX);
    if (tiles4 >= 152)
        return conv_launch_rows<CIP, COP, 4>(x, n, h, w, wt, bias, relu, y, out_f32, creal, gate, 152 * 2, st);
    return conv_launch_rows<CIP, COP, 1>(x, n, h, w, wt, bias, relu, y, out_f32, creal, gate, 152 * 8, st);
}

template <int CIP, int COP>
static cudaError_t wgrad_launch(const void* x, const void* dp, int n, int h, int w, int nslot, float* partial,
                                float* bpart, cudaStream_t st)
{
    dim3 grid(nslot, 3);
    constexpr size_t smem = wgrad_smem<CIP, COP>();
    cudaFuncSetAttribute(k_wgrad<CIP, COP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const bool vec = ((((uintptr_t)x) | ((uintptr_t)dp)) & 15) == 0;
    launch_dep(k_wgrad<CIP, COP>, grid, dim3(6 * COP), smem, st, reinterpret_cast<const bf16*>(x),
               reinterpret_cast<const bf16*>(dp), n * h, h, w, nslot, vec, partial, bpart);
    return cudaGetLastError();
}

#define GP_CNN_PAIRS(X) X(16, 32) X(32, 48) X(48, 48) X(48, 32) X(32, 32) X(32, 16)

bool cnn_pair_supported(int cip, int cop)
{
#define GP_P(a, b) if (cip == a && cop == b) return true;
    GP_CNN_PAIRS(GP_P)
#undef GP_P
    return false;
}

cudaError_t launch_cnn_conv(const void* x, int n, int h, int w, int cip, const void* wt, const float* bias, int cop,
                            int relu, void* y, int out_f32, int creal, const void* gate, cudaStream_t st)
{
#define GP_P(a, b) if (cip == a && cop == b) return conv_launch<a, b>(x, n, h, w, wt, bias, relu, y, out_f32, creal, gate, st);
    GP_CNN_PAIRS(GP_P)
#undef GP_P
    return cudaErrorInvalidValue;
}

cudaError_t launch_cnn_wgrad(const void* x, const void* dp, int n, int h, int w, int cip, int cop, int cir, int cor,
                             int nslot, float* partial, float* bpart, float* dw, float* db, cudaStream_t st)
{
    cudaError_t e = cudaErrorInvalidValue;
#define GP_P(a, b) if (cip == a && cop == b) e = wgrad_launch<a, b>(x, dp, n, h, w, nslot, partial, bpart, st);
    GP_CNN_PAIRS(GP_P)
#undef GP_P
    if (e != cudaSuccess) return e;
    launch_dep(k_wgrad_reduce, dim3((9 * cop * cip + 31) / 32 + (cop + 31) / 32), dim3(32 * WR_PARTS), 0, st, partial, bpart, nslot, cip,
               cop, cir, cor, dw, db);
    return cudaGetLastError();
}

cudaError_t launch_cnn_relu_backward(const void* dy, const void* y, void* dp, int64_t count, cudaStream_t st)
{
    const bool vec = ((((uintptr_t)dy) | ((uintptr_t)y) | ((uintptr_t)dp)) & 15) == 0;
    launch_dep(k_relu_backward, dim3(152 * 8), dim3(256), 0, st, reinterpret_cast<const bf16*>(dy),
               reinterpret_cast<const bf16*>(y), reinterpret_cast<bf16*>(dp), vec ? count / 8 : 0, count);
    return cudaGetLastError();
}

cudaError_t launch_cnn_mse(const float* pred, const float* target, int64_t npos, int cop, void* dy, float* part,
                           int nblocks, float* loss, cudaStream_t st)
{
    launch_dep(k_mse, dim3(nblocks), dim3(256), 0, st, pred, target, npos, cop, reinterpret_cast<bf16*>(dy), part);
    launch_dep(k_mse_reduce, dim3(1), dim3(32), 0, st, part, nblocks, npos, loss);
    return cudaGetLastError();
}

cudaError_t launch_cnn_pack(const float* W, const float* b, int cir, int cor, int cip, int cop, void* wt, void* wtd,
                            float* bias_p, cudaStream_t st)
{
    const int total = cop * 9 * cip;
    launch_dep(k_pack, dim3((total + 255) / 256), dim3(256), 0, st, W, b, cir, cor, cip, cop,
               reinterpret_cast<bf16*>(wt), reinterpret_cast<bf16*>(wtd), bias_p);
    return cudaGetLastError();
}

static AdamW adamw_of(float lr, float b1, float b2, float eps, int step)
{
    return {lr, b1, b2, eps, 1.f - powf(b1, (float)step), 1.f - powf(b2, (float)step)};
}

cudaError_t launch_cnn_adamw(float* p, const float* g, float* m, float* v, int64_t n, float lr, float b1, float b2,
                             float eps, float wd, int step, cudaStream_t st)
{
    launch_dep(k_adamw, dim3(152 * 2), dim3(256), 0, st, p, g, m, v, n, adamw_of(lr, b1, b2, eps, step), wd);
    return cudaGetLastError();
}

cudaError_t launch_cnn_update(const gp_cnn_layer* layers, int nlayer, float lr, float b1, float b2, float eps, float wd,
                              int step, cudaStream_t st)
{
    for (int l0 = 0; l0 < nlayer; l0 += CNN_LAYERS) {
        CnnLayers L = {};
        const int k = nlayer - l0 < CNN_LAYERS ? nlayer - l0 : CNN_LAYERS;
        int most = 0;
        for (int l = 0; l < k; ++l) {
            L.l[l] = layers[l0 + l];
            const int n = L.l[l].cin * L.l[l].cout * 9;
            most = n > most ? n : most;
        }
        launch_dep(k_update, dim3((most + 255) / 256 + 1, k), dim3(256), 0, st, L, adamw_of(lr, b1, b2, eps, step), wd);
    }
    return cudaGetLastError();
}

cudaError_t launch_cnn_features(const float* quant, int nframes, int nbox, void* feat, float* norm, cudaStream_t st)
{
    launch_dep(k_features, dim3(nframes), dim3(FEAT_NT), 0, st, quant, nbox, reinterpret_cast<bf16*>(feat), norm);
    return cudaGetLastError();
}

cudaError_t launch_cnn_denorm(const float* out, const float* norm, int nbox, int nframes, float* bkg, float* rms,
                              cudaStream_t st)
{
    const int64_t total = (int64_t)nbox * nframes;
    launch_dep(k_denorm, dim3((int)((total + 255) / 256 < 1024 ? (total + 255) / 256 : 1024)), dim3(256), 0, st, out,
               norm, nbox, total, bkg, rms);
    return cudaGetLastError();
}

cudaError_t launch_cnn_targets(const float* bkg, const float* rms, const float* norm, int nbox, int nframes,
                               float* tgt, cudaStream_t st)
{
    const int64_t total = (int64_t)nbox * nframes;
    launch_dep(k_targets, dim3((int)((total + 255) / 256 < 1024 ? (total + 255) / 256 : 1024)), dim3(256), 0, st,
               bkg, rms, norm, nbox, total, tgt);
    return cudaGetLastError();
}

}  // namespace gp
