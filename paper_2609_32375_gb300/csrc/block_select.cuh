// block_select.cuh -- exact order statistics of float32 values held across a
// thread block, without sorting them.  Used by the float32 box statistics
// (paper Section 3.1) and the learned background's feature scaling.
#pragma once
#include <stdint.h>

namespace gp {

// Unsigned integers in the order of the floats (numerically equal zeros are
// made equal first; NaN must not be passed).
__device__ __forceinline__ uint32_t key_of(float f)
{
    const uint32_t u = __float_as_uint(f + 0.f);
    return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t k)
{
    return __uint_as_float(k ^ ((k >> 31) ? 0x80000000u : 0xffffffffu));
}

constexpr int SEL_BPT = 8;        // histogram bins per thread

// Shared memory of one selection; hist is SEL_BPT * NT counters.
template <int NT>
struct SelShared {
    uint32_t hist[SEL_BPT * NT];
    uint32_t wsum[NT / 32];
    uint32_t bin, excl, cnt, next;
};

// The key of rank r (0-based) among the n keys in [klo, khi] that the block's
// threads hold, and the key of rank r + 1 in *next when `next` is given (and
// r + 1 < n).  each(f) calls f(key) for every key the calling thread holds;
// keys outside [klo, khi] are passed over.  Every thread gets the result.
//
// A pass counts the keys in SEL_BPT * NT equal bins over [klo, khi] and goes
// on inside the bin that holds rank r, until a bin is a single key.  The bins
// are taken over the range that is left, not over fixed digits, so the values
// of one sky level (whose leading bits agree) still spread over the bins:
// sky of a few hundred counts takes two passes.  At most 4 passes for 32 bits.
template <int NT, class Each>
__device__ uint32_t block_select(Each each, uint32_t klo, uint32_t khi, uint32_t r, uint32_t* next, SelShared<NT>& S)
{
    constexpr int NB = SEL_BPT * NT;
    constexpr int LB = NB >= 8192 ? 13 : NB >= 4096 ? 12 : NB >= 2048 ? 11 : 10;   // log2 NB
    static_assert(NB == 1 << LB, "a power of two of bins");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t equal = 0;
    const bool whole = klo == khi;
    while (klo != khi) {
        const int bits = 32 - __clz(khi - klo);
        const int shift = bits > LB ? bits - LB : 0;
        for (int b = tid; b < NB; b += NT) S.hist[b] = 0u;
        __syncthreads();
        each([&](uint32_t k) {
            if (k >= klo && k <= khi) atomicAdd(&S.hist[(k - klo) >> shift], 1u);
        });
        __syncthreads();
        uint32_t c[SEL_BPT], tot = 0;
#pragma unroll
        for (int q = 0; q < SEL_BPT / 4; ++q) {
            const uint4 h = reinterpret_cast<const uint4*>(S.hist)[tid * (SEL_BPT / 4) + q];
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
        uint32_t base = 0;
        for (int w = 0; w < warp; ++w) base += S.wsum[w];
        uint32_t excl = base + incl - tot;
        if (r >= excl && r < excl + tot) {
            uint32_t bin = 0, cnt = c[0];
#pragma unroll
            for (int q = 1; q < SEL_BPT; ++q)
                if (bin == q - 1 && r >= excl + c[q - 1]) {
                    excl += c[q - 1];
                    bin = q;
                    cnt = c[q];
                }
            S.bin = tid * SEL_BPT + bin;
            S.excl = excl;
            S.cnt = cnt;
        }
        __syncthreads();
        r -= S.excl;
        equal = S.cnt;
        klo += S.bin << shift;
        const uint32_t top = klo + ((1u << shift) - 1u);
        khi = top < khi ? top : khi;
    }
    if (next) {
        // still inside the run of equal keys, or the smallest larger key
        if (whole || r + 1 < equal) {
            *next = klo;
        } else {
            if (tid == 0) S.next = 0xffffffffu;
            __syncthreads();
            uint32_t m = 0xffffffffu;
            each([&](uint32_t k) { if (k > klo && k < m) m = k; });
            m = __reduce_min_sync(0xffffffffu, m);
            if (lane == 0) atomicMin(&S.next, m);
            __syncthreads();
            *next = S.next;
        }
    }
    return klo;
}

}  // namespace gp
