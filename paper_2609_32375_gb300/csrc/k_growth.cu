// k_growth.cu -- growth curves by top-hat apertures (paper Section 3.4):
// for each source and each integer radius r of a list, the sum of m = I - B
// over the top-hat {(u, v) : u^2 + v^2 <= r^2} centred on the pixel nearest
// the source, (floor(x + 1/2), floor(y + 1/2)), with sigma^2 summed over the
// same pixels -- the value at that pixel of the frame's cross-correlation
// with the top-hat, which the paper evaluates by FFT for all pixels at once.
// Here only the sources' pixels are visited.
//
// One warp per source, a lane per column of the largest top-hat, rows in
// order.  Every pixel is added once, to the ring of radii it opens: the
// smallest r_k with r_k^2 >= u^2 + v^2 (a table over u^2 + v^2).  A lane
// keeps float-float sums for its current ring and adds them into its
// slot for that ring in shared memory when the ring changes (down a column
// the ring index falls, then rises: at most two stretches per ring).  Then
// lane k sums ring k's 32 slots in lane order, and a scan across the lanes turns
// ring sums into the growth curve (radius k = rings 0..k).  Fixed orders
// throughout: the sums are reproducible.
//
// A source whose window lies inside the frame and in one or two intervals of
// the background mesh's rows (most do) takes its pixels ring by ring instead, 32
// at a time from a list made on the host: every lane has a pixel, a
// ring's sums are written once, and the column and row terms of the splines
// come from shared memory.  Bound by instruction issue: 15,000 sources of 13
// radii (3..15) take 120 us, 154 by columns (6,300 warp instructions a
// source, much of it lanes changing rings at different rows) and 188 before
// that, with the row coefficients divided out by every lane.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "gp_internal.cuh"
#include "gp_launch.h"

namespace gp {

constexpr int GR_NT = 128;                 // 4 warps per CTA
constexpr int GR_W = GR_NT / 32;
constexpr int GR_ROWS = 4;                 // rows of pixels loaded ahead

// most list entries (pixels of the largest top-hat, each ring rounded up to
// 32) of the ring-by-ring form: radii up to about 35
constexpr int GR_LIST = 4096;
constexpr int GR_NONE = 0x7f;              // u of an empty entry

// the ring lists: u | v << 8 (bytes), ring after ring, and the ring of each 32
struct GrowthList {
    alignas(16) uint16_t uv[GR_LIST];      // (read by words)
    int8_t ring[GR_LIST / 32];
};

struct GrowthSpec {
    int list;                   // entries of the ring lists (0: the column form only)
    int nr;
    int r[GP_GROWTH_MAX_NR];
    int rmax;
    float gain;
    double inv_gain;            // 1 / gain (0 when gain <= 0)
};

// dynamic shared memory: the ring table (int8 per u^2 + v^2 up to rmax^2),
// then per warp: flux and variance slots [32 lanes][S] (float-float) and flag
// slots [32][S] (bytes), S = nr rounded up to odd so that lane k reading ring k of
// every lane meets no bank conflict
template <bool F32>
__global__ void __launch_bounds__(GR_NT) k_growth(Image im, SplineTab sb, SplineTab sr,
                                                  const __grid_constant__ GrowthSpec gs,
                                                  const __grid_constant__ GrowthList gl, const double* __restrict__ xs,
                                                  const double* __restrict__ ys, int n, const int* __restrict__ n_dev,
                                                  double* flux, double* ferr, uint32_t* flags)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int nr = gs.nr, rmax = gs.rmax, r2max = rmax * rmax;
    int8_t* ring_of = reinterpret_cast<int8_t*>(smem);
    const size_t tab = ((size_t)r2max + 1 + 15) & ~(size_t)15;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int S = nr | 1, NS = 32 * S;
    float2* sf = reinterpret_cast<float2*>(smem + tab) + (size_t)warp * NS * 2;
    float2* sv = sf + NS;
    uint8_t* sfl = smem + tab + (size_t)GR_W * NS * 2 * sizeof(float2) + (size_t)warp * NS;
    // per warp the columns' spline terms for two intervals of the mesh's rows
    // and the rows' terms (80 bytes for each of side); the ring lists
    const int side = 2 * rmax + 1;
    unsigned char* more = smem + tab + (size_t)GR_W * NS * (2 * sizeof(float2) + 1);
    ulonglong2* colt = reinterpret_cast<ulonglong2*>(more) + (size_t)warp * 5 * side;          // [2][side][2]
    float4* rowt = reinterpret_cast<float4*>(colt + 4 * side);
    uint16_t* off = reinterpret_cast<uint16_t*>(reinterpret_cast<ulonglong2*>(more) + (size_t)GR_W * 5 * side);
    int8_t* oring = reinterpret_cast<int8_t*>(off + gs.list);
    for (int i = threadIdx.x; i < gs.list / 2; i += GR_NT)
        reinterpret_cast<uint32_t*>(off)[i] = reinterpret_cast<const uint32_t*>(gl.uv)[i];
    for (int i = threadIdx.x; i < gs.list / 32; i += GR_NT) oring[i] = gl.ring[i];
    for (int d2 = threadIdx.x; d2 <= r2max; d2 += GR_NT) {
        int k = 0;
        while (k < nr && gs.r[k] * gs.r[k] < d2) ++k;
        ring_of[d2] = (int8_t)k;                        // k < nr: every d2 <= rmax^2 opens some radius
    }
    __syncthreads();
    const int nstep = gs.list / 32;
    const int W = im.W, H = im.H;
    const int wid = blockIdx.x * GR_W + warp, nw = gridDim.x * GR_W;
    if (n_dev) n = min(n, *n_dev);           // a device count (catalog rows), at most n
    for (int s = wid; s < n; s += nw) {
        const double cxd = xs[s] + 0.5, cyd = ys[s] + 0.5;
        // positions far outside the frame (or NaN) give empty sums, flagged
        const bool near = fabsf((float)cxd - 0.5f * W) <= 0.5f * W + 4096.f && fabsf((float)cyd - 0.5f * H) <= 0.5f * H + 4096.f;
        const int xc = near ? __double2int_rd(cxd) : -(1 << 20), yc = near ? __double2int_rd(cyd) : -(1 << 20);
        // the intervals of the mesh's rows at the first and the last row
        const bool inside = nstep && near && xc >= rmax && xc + rmax < W && yc >= rmax && yc + rmax < H;
        const int j0 = inside ? axis_coef(sb.ay, (float)(yc - rmax)).i : 0;
        const int jn = inside ? axis_coef(sb.ay, (float)(yc + rmax)).i - j0 : 2;
        if (jn <= 1) {
            for (int q = lane; q < side; q += 32) {
                const AxCoef cx = axis_coef(sb.ax, (float)(xc - rmax + q)), cy = axis_coef(sb.ay, (float)(yc - rmax + q));
                float2 b0 = row_eval(sb, j0, cx), r0 = row_eval(sr, j0, cx);
                for (int t = 0; t <= jn; ++t) {
                    const int j1 = min(j0 + t + 1, sb.ay.n - 1);
                    const float2 b1 = row_eval(sb, j1, cx), r1 = row_eval(sr, j1, cx);
                    const unsigned long long u0 = f2pack(b0.x, r0.x);
                    ulonglong2* c = colt + 2 * (t * side + q);
                    c[0] = make_ulonglong2(u0, f2sub(f2pack(b1.x, r1.x), u0));
                    c[1] = make_ulonglong2(f2pack(b0.y, r0.y), f2pack(b1.y, r1.y));
                    b0 = b1;
                    r0 = r1;
                }
                rowt[q] = make_float4(cy.b, cy.c0, cy.c1, __int_as_float(2 * side * (cy.i - j0)));
            }
            __syncwarp();
            DF2 cs;
            cs.hi = cs.lo = 0ull;
            uint32_t cfl = 0u;
            for (int t0 = 0; t0 < nstep; t0 += GR_ROWS) {
                int o[GR_ROWS];
                float val[GR_ROWS];
                bool bad[GR_ROWS];
#pragma unroll
                for (int j = 0; j < GR_ROWS; ++j) {
                    o[j] = t0 + j < nstep ? off[(t0 + j) * 32 + lane] : GR_NONE;
                    val[j] = 0.f;
                    bad[j] = false;
                    if (o[j] != GR_NONE) val[j] = load_px<F32>(im, xc + (int8_t)(o[j] & 0xff), yc + (int8_t)(o[j] >> 8), bad[j]);
                }
#pragma unroll
                for (int j = 0; j < GR_ROWS; ++j) {
                    if (t0 + j >= nstep) break;
                    if (o[j] != GR_NONE) {
                        const int u = (int8_t)(o[j] & 0xff) + rmax, v = (int8_t)(o[j] >> 8) + rmax;
                        const float4 rc = rowt[v];
                        const ulonglong2* cu = colt + 2 * u + __float_as_int(rc.w);
                        const ulonglong2 c0 = cu[0], c1 = cu[1];
                        // axis_combine of both maps
                        const unsigned long long bs =
                            f2fma(f2pack(rc.z, rc.z), c1.y, f2fma(f2pack(rc.y, rc.y), c1.x, f2fma(f2pack(rc.x, rc.x), c0.y, c0.x)));
                        const float m = val[j] - f2lo(bs), sg = f2hi(bs);
                        if (bad[j]) {
                            cfl |= GP_FLAG_BAD;
                        } else {
                            if (im.sat > 0.f && val[j] >= im.sat) cfl |= GP_FLAG_SAT;
                            const float p = sg * sg;
                            df2_add(cs, f2pack(m, p));
                            cs.lo = f2add(cs.lo, f2pack(0.f, fmaf(sg, sg, -p)));
                        }
                    }
                    const int k = oring[t0 + j];
                    if (t0 + j + 1 == nstep || oring[t0 + j + 1] != k) {     // the ring's last pixels
                        const int q = lane * S + k;
                        sf[q] = make_float2(f2lo(cs.hi), f2lo(cs.lo));
                        sv[q] = make_float2(f2hi(cs.hi), f2hi(cs.lo));
                        sfl[q] = (uint8_t)cfl;
                        cs.hi = cs.lo = 0ull;
                        cfl = 0u;
                    }
                }
            }
            __syncwarp();
        } else {
        for (int i = lane; i < NS; i += 32) {
            sf[i] = make_float2(0.f, 0.f);
            sv[i] = make_float2(0.f, 0.f);
            sfl[i] = 0u;
        }
        __syncwarp();
        for (int u0 = -rmax; u0 <= rmax; u0 += 32) {
            const int u = u0 + lane;
            const bool col = u <= rmax;
            const int x = xc + u;
            const bool xin = x >= 0 && x < W;
            const AxCoef ccx = axis_coef(sb.ax, (float)(xin ? x : 0));
            int jc = -1;
            // both maps of the column, (background, noise) in a pair: values
            // and their differences between the two node rows, second derivatives
            unsigned long long u_0 = 0, u_d = 0, w_0 = 0, w_1 = 0;
            int kc = -1;
            DF2 cs;                                     // (sum of m, sum of sigma^2)
            cs.hi = cs.lo = 0ull;
            uint32_t cfl = 0u;
            auto flush = [&]() {
                if (kc >= 0) {
                    const int q = lane * S + kc;
                    DF a, c;
                    a.hi = sf[q].x; a.lo = sf[q].y;
                    c.hi = f2lo(cs.hi); c.lo = f2lo(cs.lo);
                    a = df_merge(a, c);
                    sf[q] = make_float2(a.hi, a.lo);
                    a.hi = sv[q].x; a.lo = sv[q].y;
                    c.hi = f2hi(cs.hi); c.lo = f2hi(cs.lo);
                    a = df_merge(a, c);
                    sv[q] = make_float2(a.hi, a.lo);
                    sfl[q] |= (uint8_t)cfl;
                }
                cs.hi = cs.lo = 0ull;
                cfl = 0u;
            };
            const int uu = u * u;
            for (int vb = -rmax; vb <= rmax; vb += 32) {
                // the coefficients of 32 rows, one a lane, fetched by shuffle
                const AxCoef cl = axis_coef(sb.ay, (float)min(max(yc + vb + lane, 0), H - 1));
                const int ve = min(rmax, vb + 31);
                for (int v0 = vb; v0 <= ve; v0 += GR_ROWS) {
                    // the rows' pixels first, so that their loads overlap
                    float val[GR_ROWS];
                    bool bad[GR_ROWS];
#pragma unroll
                    for (int j = 0; j < GR_ROWS; ++j) {
                        const int v = v0 + j, y = yc + v;
                        val[j] = 0.f;
                        bad[j] = false;
                        if (col && v <= ve && uu + v * v <= r2max && xin && (unsigned)y < (unsigned)H)
                            val[j] = load_px<F32>(im, x, y, bad[j]);
                    }
#pragma unroll
                    for (int j = 0; j < GR_ROWS; ++j) {
                        const int v = v0 + j;
                        if (v > ve) break;                        // the whole warp
                        const int yi = __shfl_sync(0xffffffffu, cl.i, v - vb);
                        const float yb = __shfl_sync(0xffffffffu, cl.b, v - vb);
                        const float y0 = __shfl_sync(0xffffffffu, cl.c0, v - vb), y1 = __shfl_sync(0xffffffffu, cl.c1, v - vb);
                        const int d2 = uu + v * v;
                        if (!col || d2 > r2max) continue;
                        const int k = ring_of[d2];
                        if (k != kc) {
                            flush();
                            kc = k;
                        }
                        if (!xin || (unsigned)(yc + v) >= (unsigned)H) {
                            cfl |= GP_FLAG_TRUNCATED;
                            continue;
                        }
                        if (bad[j]) {
                            cfl |= GP_FLAG_BAD;
                            continue;
                        }
                        if (yi != jc) {
                            const int yi1 = min(yi + 1, sb.ay.n - 1);
                            const float2 b0 = row_eval(sb, yi, ccx), b1 = row_eval(sb, yi1, ccx);
                            const float2 r0 = row_eval(sr, yi, ccx), r1 = row_eval(sr, yi1, ccx);
                            u_0 = f2pack(b0.x, r0.x);
                            u_d = f2sub(f2pack(b1.x, r1.x), u_0);
                            w_0 = f2pack(b0.y, r0.y);
                            w_1 = f2pack(b1.y, r1.y);
                            jc = yi;
                        }
                        // axis_combine of both maps
                        const unsigned long long bs =
                            f2fma(f2pack(y1, y1), w_1, f2fma(f2pack(y0, y0), w_0, f2fma(f2pack(yb, yb), u_d, u_0)));
                        const float m = val[j] - f2lo(bs), sg = f2hi(bs);
                        if (im.sat > 0.f && val[j] >= im.sat) cfl |= GP_FLAG_SAT;
                        // m, and sigma^2 as its product and the product's rounding error
                        const float p = sg * sg;
                        df2_add(cs, f2pack(m, p));
                        cs.lo = f2add(cs.lo, f2pack(0.f, fmaf(sg, sg, -p)));
                    }
                }
            }
            flush();
            __syncwarp();
        }
        }
        // ring sums over the lanes in order (lane groups share a ring's lanes
        // when there are few rings), then radius k = rings 0..k (a scan whose
        // combination order is fixed)
        DF rf = df_zero(), rv = df_zero();
        uint32_t rfl = 0u;
        const int per = nr <= 8 ? 8 : nr <= 16 ? 16 : 32, ring = lane & (per - 1);
        if (ring < nr) {
            for (int l = lane & ~(per - 1), e = l + per; l < e; ++l) {
                const int q = l * S + ring;
                DF a;
                a.hi = sf[q].x; a.lo = sf[q].y;
                rf = df_merge(rf, a);
                a.hi = sv[q].x; a.lo = sv[q].y;
                rv = df_merge(rv, a);
                rfl |= sfl[q];
            }
        }
        for (int o = per; o < 32; o <<= 1) {
            DF pf, pv;
            pf.hi = __shfl_xor_sync(0xffffffffu, rf.hi, o); pf.lo = __shfl_xor_sync(0xffffffffu, rf.lo, o);
            pv.hi = __shfl_xor_sync(0xffffffffu, rv.hi, o); pv.lo = __shfl_xor_sync(0xffffffffu, rv.lo, o);
            rf = df_merge(rf, pf);
            rv = df_merge(rv, pv);
            rfl |= __shfl_xor_sync(0xffffffffu, rfl, o);
        }
        if (lane >= nr) {
            rf = rv = df_zero();
            rfl = 0u;
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            DF pf, pv;
            pf.hi = __shfl_up_sync(0xffffffffu, rf.hi, o); pf.lo = __shfl_up_sync(0xffffffffu, rf.lo, o);
            pv.hi = __shfl_up_sync(0xffffffffu, rv.hi, o); pv.lo = __shfl_up_sync(0xffffffffu, rv.lo, o);
            const uint32_t pfl = __shfl_up_sync(0xffffffffu, rfl, o);
            if (lane >= o) {
                rf = df_merge(pf, rf);
                rv = df_merge(pv, rv);
                rfl |= pfl;
            }
        }
        if (lane < nr) {
            const double F = df_value(rf);
            double V = df_value(rv);
            if (gs.gain > 0.f && F > 0.0) V = fma(F, gs.inv_gain, V);
            const int64_t o = (int64_t)s * nr + lane;
            flux[o] = F;
            ferr[o] = V > 0.0 ? sqrt(V) : 0.0;
            flags[o] = rfl;
        }
        __syncwarp();
    }
}

static size_t growth_smem_bytes(int nr, int rmax, int list)
{
    const size_t tab = ((size_t)rmax * rmax + 1 + 15) & ~(size_t)15, side = 2 * (size_t)rmax + 1;
    size_t b = tab + (size_t)GR_W * (nr | 1) * 32 * (2 * sizeof(float2) + 1);
    if (list) b += GR_W * side * 80 + (size_t)list * 2 + list / 32;
    return (b + 15) & ~(size_t)15;
}

cudaError_t launch_growth(const Image& im, const SplineTab& sb, const SplineTab& sr, const double* xs,
                          const double* ys, int n, const int* n_dev, const int* radii, int nr, float gain,
                          double* flux, double* ferr, uint32_t* flags, cudaStream_t st)
{
    GrowthSpec gs;
    memset(&gs, 0, sizeof gs);
    gs.nr = nr;
    for (int k = 0; k < nr; ++k) gs.r[k] = radii[k];
    gs.rmax = radii[nr - 1];
    gs.gain = gain;
    gs.inv_gain = gain > 0.f ? 1.0 / (double)gain : 0.0;
    GrowthList gl;
    constexpr int RMAX_LIST = 36;            // a disc of radius 37 alone has more than GR_LIST pixels
    if (gs.rmax <= RMAX_LIST) {
        int cnt[GP_GROWTH_MAX_NR] = {}, at[GP_GROWTH_MAX_NR], ring[RMAX_LIST * RMAX_LIST + 1], total = 0;
        for (int d2 = 0, k = 0; d2 <= gs.rmax * gs.rmax; ++d2) {
            while (gs.r[k] * gs.r[k] < d2) ++k;
            ring[d2] = k;
        }
        auto each = [&](auto f) {
            for (int v = -gs.rmax; v <= gs.rmax; ++v)
                for (int u = -gs.rmax; u <= gs.rmax; ++u)
                    if (u * u + v * v <= gs.rmax * gs.rmax) f(ring[u * u + v * v], u, v);
        };
        each([&](int k, int, int) { ++cnt[k]; });
        for (int k = 0; k < nr; ++k) {
            at[k] = total;
            total += (cnt[k] + 31) & ~31;
        }
        if (total <= GR_LIST) {
            gs.list = total;
            for (int i = 0; i < total; ++i) gl.uv[i] = GR_NONE;
            for (int k = 0; k < nr; ++k)
                for (int i = at[k]; i < at[k] + cnt[k]; i += 32) gl.ring[i / 32] = (int8_t)k;
            each([&](int k, int u, int v) { gl.uv[at[k]++] = (uint16_t)((u & 0xff) | (v & 0xff) << 8); });
        }
    }
    const size_t smem = growth_smem_bytes(nr, gs.rmax, gs.list);
    const int grid = 152 * std::max(1, std::min(6, (int)(220 * 1024 / (smem + 1024))));   // as many as fit an SM
    if (im.is_f32) {
        cudaFuncSetAttribute(k_growth<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_growth<true><<<grid, GR_NT, smem, st>>>(im, sb, sr, gs, gl, xs, ys, n, n_dev, flux, ferr, flags);
    } else {
        cudaFuncSetAttribute(k_growth<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_growth<false><<<grid, GR_NT, smem, st>>>(im, sb, sr, gs, gl, xs, ys, n, n_dev, flux, ferr, flags);
    }
    return cudaGetLastError();
}

}  // namespace gp
