// k_stream.cu -- launch of the streaming detection pass (k_stream_impl.cuh:
// spline background and noise, matched filter, threshold, packed mask, zero
// map and the list of detection tiles with foreground; paper Section 3.2 with
// the Section 3.1 maps) and its form for a caller's mask (k_pack_mask, for
// gp_label_mask).
#include <stdlib.h>
#include <string.h>

#include <algorithm>

#include "k_stream_impl.cuh"

namespace gp {

cudaError_t launch_stream_u16(const DetectArgs* args, const DetectArgs* batch, int nframes, bool fast,
                              const CUtensorMap* maps, cudaStream_t st);
cudaError_t launch_stream_f32(const DetectArgs* args, const DetectArgs* batch, int nframes, bool fast,
                              const CUtensorMap* maps, cudaStream_t st);

// ------------------------------------------------------- given masks ---
// gp_label_mask: the caller's byte mask packed into the same bit layout,
// with the zero map and the tile list (one warp per strip and tile band)
template <bool BATCH>
__global__ void __launch_bounds__(128) k_pack_mask(const DetectArgs* __restrict__ batch,
                                                   const __grid_constant__ DetectArgs one)
{
    const DetectArgs& A = stream_args<BATCH>(batch, one);
    const int W = A.im.W, Hf = A.im.H;
    const int lane = threadIdx.x & 31;
    const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nty = (Hf + TY - 1) / TY;
    if (wid >= A.nstrip * nty) return;
    const int strip = wid % A.nstrip, ty = wid / A.nstrip;
    const int xs = strip * ST_STRIP + ST_CPL * lane;
    uint32_t orw = 0u;
    for (int y = ty * TY; y < min(Hf, ty * TY + TY); ++y) {
        bool fg[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const bool in = xs + e < W;
            fg[e] = in && A.in_mask[(int64_t)y * W + xs + e] != 0;
            if (in) A.seg[(int64_t)y * W + xs + e] = 0u;
        }
        const uint32_t b0 = __ballot_sync(0xffffffffu, fg[0]), b1 = __ballot_sync(0xffffffffu, fg[1]);
        const uint32_t b2 = __ballot_sync(0xffffffffu, fg[2]), b3 = __ballot_sync(0xffffffffu, fg[3]);
        orw |= b0 | b1 | b2 | b3;
        if (lane == 0) A.bits[(int64_t)y * A.nstrip + strip] = make_uint4(b0, b1, b2, b3);
    }
    if (lane < 2) {
        const int tcol = 2 * strip + lane;
        if (tcol < A.T.ntx) {
            const int tile = ty * A.T.ntx + tcol;
            if (orw & (lane ? 0xffff0000u : 0x0000ffffu)) A.tl_list[atomicAdd(A.tl_count, 1)] = tile;
            else A.T.piece_cnt[tile] = 0;
        }
    }
}

// ------------------------------------------------------------ launchers ---
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

static int stream_force_direct = -1;   // GP_STREAM_DIRECT=1 in the environment: the DIRECT staging everywhere

// a tensor map of the frame for G-row groups, or false when the frame's rows
// are not 16-byte aligned (or the frame is too small for the mirror rows)
static bool make_tmap(const Image& im, int G, CUtensorMap* map)
{
    if (stream_force_direct < 0) {
        const char* e = getenv("GP_STREAM_DIRECT");
        stream_force_direct = (e && e[0] == '1') ? 1 : 0;
    }
    if (stream_force_direct) return false;
    const int esz = im.is_f32 ? 4 : 2;
    if (im.mask) return false;
    if (im.W < 2 * ST_HALO || im.H < 2 * ST_HALO) return false;
    if ((((uintptr_t)im.data) & 15) || ((im.pitch * esz) & 15)) return false;
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {(cuuint64_t)im.W, (cuuint64_t)im.H};
    cuuint64_t strides[1] = {(cuuint64_t)(im.pitch * esz)};
    cuuint32_t box[2] = {(cuuint32_t)ST_BOXW, (cuuint32_t)G};
    cuuint32_t es[2] = {1, 1};
    const CUresult r = fn(map, im.is_f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16, 2,
                          const_cast<void*>(im.data), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

static int pack_warps(int W, int H) { return ((W + ST_STRIP - 1) / ST_STRIP) * ((H + TY - 1) / TY); }

// rows per group of the streaming pass for a padded kernel size
static int stream_group_rows(int ks)
{
    switch (ks) {
    case 3: return StreamCfg<3>::G;
    case 5: return StreamCfg<5>::G;
    case 7: return StreamCfg<7>::G;
    default: return StreamCfg<15>::G;
    }
}

// the padded kernel size the streaming pass runs for a kw x kh kernel
int stream_ks(int kw, int kh)
{
    const int k = kw > kh ? kw : kh;
    return k <= 3 ? 3 : k <= 5 ? 5 : k <= 7 ? 7 : 15;
}

int stream_ctas(int W, int H, int rows)
{
    return ((W + ST_COLS - 1) / ST_COLS) * ((H + rows - 1) / rows);
}

// Output rows per CTA.  A CTA takes about as long as its row groups, alone on
// an SM or with as many others as fit (four for 3 and 5 taps by tensor maps,
// down to one for 15 taps of float32), so the pass lasts its waves of resident
// x 152 CTAs times the groups of one, and 1.5 more for filling the pipeline.
// Shorter CTAs read and filter more halo rows (8 groups of 5 for 32 rows, 27
// for 128).  1 MP float32, 5 taps: 85 us at 128 rows, 33 at 32; 4 MP uint16: 75
// and 32; 17 MP float32: 92 and 64 (64 rows).
int stream_rows(const DetectArgs* args, int n, int G, int resident)
{
    int best = ST_RC;
    double least = 0.0;
    for (int rows = ST_RC; rows >= TY; rows >>= 1) {
        int64_t ctas = 0;
        for (int f = 0; f < n; ++f) ctas += stream_ctas(args[f].im.W, args[f].im.H, rows);
        const int groups = (rows + 2 * (args[0].ks / 2) + G - 1) / G, wave = resident * 152;
        const double t = (double)((ctas + wave - 1) / wave) * (groups + 1.5);
        if (rows == ST_RC || t < least) {
            least = t;
            best = rows;
        }
    }
    return best;
}

cudaError_t launch_stream_any(const DetectArgs* args, const DetectArgs* batch, int nframes, cudaStream_t st)
{
    const DetectArgs& one = args[0];
    if (one.in_mask) {
        int warps = 0;
        for (int f = 0; f < nframes; ++f) warps = std::max(warps, pack_warps(args[f].im.W, args[f].im.H));
        const int blocks = (warps + 3) / 4;
        if (batch) k_pack_mask<true><<<dim3(blocks, nframes), 128, 0, st>>>(batch, one);
        else k_pack_mask<false><<<blocks, 128, 0, st>>>(nullptr, one);
        return cudaGetLastError();
    }
    const int G = stream_group_rows(one.ks);
    CUtensorMap maps[MAX_BATCH];
    bool fast = one.nrank == 1 && one.ks <= 7, tma = true;
    for (int f = 0; f < nframes; ++f) {
        const DetectArgs& A = args[f];
        fast = fast && !A.mask_out && !A.nnear && !A.im.mask;
        tma = tma && make_tmap(A.im, G, maps + f);
    }
    const CUtensorMap* mp = tma ? maps : nullptr;
    if (one.im.is_f32) return launch_stream_f32(args, batch, nframes, fast, mp, st);
    return launch_stream_u16(args, batch, nframes, fast, mp, st);
}

}  // namespace gp
