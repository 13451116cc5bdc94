// k_deblend.cu -- multi-threshold deblending of the segments (the
// SExtractor reading of the detection; the paper's own detection takes local
// maxima).  For a segment S of at least 2 minarea pixels, with
// nu = F / sigma its significance:
//  - levels t_i = k (nu_max / k)^(i / N), i = 0..N-1, with k the detection
//    threshold and nu_max the segment's peak;
//  - the branches of level i are the 8-connected components of
//    {p in S : nu(p) > t_i} (level 0: S itself);
//  - a branch is significant when it has minarea pixels and its sum of m
//    exceeds mincont times the segment's (the segment's sum must be > 0);
//  - from the root up: a branch passes on to its significant children (two
//    or more: a split, each examined in turn; one: it continues there); a
//    branch without one is a seed;
//  - with two or more seeds the other pixels are attributed by growth from
//    the seeds within the level sets, from the highest level down: in rounds,
//    an unattributed pixel of the level set takes the smallest seed rank
//    among its attributed 8-neighbours (ranks in the order of the seeds'
//    first pixels); the objects are labelled 1 + their minimum linear index.
//
// A team of threads per candidate segment, its bounding box in global
// scratch: a warp for boxes up to DB_SMALL pixels (more in crowded frames), a group of DB_GW warps up to
// DB_MED, a CTA above, a cluster of 8 CTAs above DB_BIG.  One launch serves all:
// its clusters first work through the big candidates together, then each CTA
// through the larger ones, each group through the middle ones and each warp
// through the small ones, all by claims on shared counters.
// The time is the largest candidate's: a nebulosity whose box holds 55,000
// pixels takes 30 levels of five passes over its pixels, then some 250 growth
// rounds, 0.96 ms in all (a single CTA took 6 to 15 ms on such a field).  The
// thousands of stars beside it are short and wait on memory and barriers, so
// many run side by side.  It hangs on the field: two crowded 17 MP frames with
// nebulosity 11.4 and 11.5 ms a call with a CTA a candidate, 1.9 and 1.7 so; the
// 151 MP frame 19.0 and 3.4; a 4 MP CCD frame without nebulosity 0.92 and 0.60.
//
// Sums of m are exact 64-bit fixed-point integers (m scaled by 2^20), the
// level sets' components come from a lock-free union-find whose roots are the
// components' minimum pixels, and the growth is synchronous, so the result
// does not depend on the order in which threads run.  The objects' catalog
// rows are formed from float64 sums in a fixed order and ranked by label.
#include <cooperative_groups.h>
#include <limits.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "gp_internal.cuh"
#include "gp_launch.h"

namespace gp {

namespace cg = cooperative_groups;

constexpr int DB_NT = 1024;                   // one CTA an SM
constexpr int DB_CL = 8;                     // CTAs of a cluster
// Box pixels: a warp's most, a group's most, a CTA's most.  The lone candidate
// of a sparse frame sets the time there, so a team is as large as its box can
// use: a warp takes 1.1 ms for a box of 1,000 pixels, a group 0.4, and the stars
// of a 300 x 257 frame 0.43 ms in groups above 128 pixels, 0.74 above 256.  A 4 MP
// CCD frame's 2,471 candidates take 0.60 ms with a warp's limit at 64 or 128
// pixels, 0.74 at 256, 1.66 at 1,024 and no groups; groups of 4 warps 0.72; CTAs
// in place of the groups 0.59, but then a crowded 17 MP field, whose groups
// number thousands, 5 % more.  64 against 128: the 162 stars of a 512 x 512 frame
// with boxes up to 100 pixels 0.30 and 0.38 ms.
// DB_BIG at 4,096 or 16,384 makes no difference to a crowded 17 MP field.
constexpr int DB_SMALL = 64, DB_MED = 1024, DB_BIG = 8192;
// a warp's most in frames with more segments than the chip has warps, where
// throughput counts (the 40,130 of a crowded 151 MP frame, 6,000 of them with
// boxes of 65 to 128 pixels: 3.74 ms with 64, 3.43 with 128, 3.37 with 256)
constexpr int DB_MANY = 32 * 152, DB_SMALL_MANY = 128;
constexpr int DB_GW = 8;                     // warps of a group
// box pixels of an object's catalog row: a warp's most (crowded 17 MP field, 256,
// 1,024 and 4,096: 1.91, 1.91 and 1.96 ms)
constexpr int DB_ROW = 1024;
// the call's counters, one 256-byte block cleared per call: candidates larger
// than DB_SMALL, staged objects, small candidates, big ones; the next big,
// CTA's, small and group's one to claim; then the first big candidates' indexes
// (any more are a CTA's)
enum {
    DBC_N = 0, DBC_OBJ = 1, DBC_SMALL = 2, DBC_BIG = 3, DBC_NEXT_BIG = 4, DBC_NEXT = 5, DBC_NEXT_SMALL = 6, DBC_NEXT_MED = 7,
    DBC_LIST = 8
};
constexpr int DB_CTL = 64, DB_MAX_BIG = DB_CTL - DBC_LIST;
constexpr int DB_MAX_SEEDS = 1024;
constexpr int DB_MAX_LEVELS = 64;            // nthresh at most (checked by the API)
constexpr double DB_FIX = 1048576.0;         // 2^20

struct DeblendArgs {
    Image im;
    SplineTab sb, sr;
    int kw, kh;
    float taps[KMAX];
    float thresh;
    int minarea, nthresh;
    double mincont;
    uint32_t* seg;
    // the catalog rows of the segments
    const int* n_dev;
    int cap;
    const uint32_t* label;
    const int* npix;
    const int *xmin, *xmax, *ymin, *ymax;
    // candidates (the larger ones from the front, a group's as ~row; the small
    // ones from the back), counters and scratch
    int* cand;
    int* ctl;
    int64_t* off;            // [cand] first scratch byte of each candidate (-1: no room)
    char* scratch;
    // objects: staging rows, then the caller's catalog in label order
    DbObj* obj;
    int* obj_count;
    int obj_stage_cap;
    int* counts;             // [2] segments split, objects
    int* status;
};

// the scratch arrays of a candidate with area A and halo area AH
struct DbScratch {
    float* mh;      // [AH] m over the box and the filter halo
    float* nu;      // [A]  nu, -1 outside the segment
    long long* mf;  // [A]  m in fixed point
    int* lab;       // [A]  union-find of the current level
    int* act;       // [A]  active node of the pixel (-1 none)
    int* seed;      // [A]  seed id + 1 (0 none)
    long long* fs;  // [A + 1] branch sums
    int* cnt;       // [A + 1] branch pixel counts; then seed ranks
    int* sig;       // [A + 1] significant branch (root) / node with a significant child
    int* own;       // [A]  object rank (0 none)
    int* own2;      // [A]
    int* first;     // [A + 1] first pixel of each seed
};

__device__ DbScratch db_scratch(char* base, int A, int AH)
{
    DbScratch s;
    char* p = base;
    auto take = [&](size_t bytes) { char* q = p; p += (bytes + 15) & ~(size_t)15; return q; };
    s.mh = reinterpret_cast<float*>(take((size_t)AH * 4));
    s.nu = reinterpret_cast<float*>(take((size_t)A * 4));
    s.mf = reinterpret_cast<long long*>(take((size_t)A * 8));
    s.lab = reinterpret_cast<int*>(take((size_t)A * 4));
    s.act = reinterpret_cast<int*>(take((size_t)A * 4));
    s.seed = reinterpret_cast<int*>(take((size_t)A * 4));
    s.fs = reinterpret_cast<long long*>(take((size_t)(A + 1) * 8));
    s.cnt = reinterpret_cast<int*>(take((size_t)(A + 1) * 4));
    s.sig = reinterpret_cast<int*>(take((size_t)(A + 1) * 4));
    s.own = reinterpret_cast<int*>(take((size_t)A * 4));
    s.own2 = reinterpret_cast<int*>(take((size_t)A * 4));
    s.first = reinterpret_cast<int*>(take((size_t)(A + 1) * 4));
    return s;
}

__host__ __device__ inline int64_t db_scratch_bytes(int64_t A, int64_t AH)
{
    auto r = [](int64_t b) { return (b + 15) & ~(int64_t)15; };
    return r(AH * 4) + r(A * 4) + r(A * 8) + 4 * r(A * 4) + r((A + 1) * 8) + 2 * r((A + 1) * 4) + r((A + 1) * 4) +
           r(A * 4);
}

__device__ int db_find(int* lab, int x)
{
    for (int n = 0; n < (1 << 24); ++n) {
        const int p = lab[x];
        if (p == x) return x;
        const int g = lab[p];
        if (g != p) lab[x] = g;
        x = g;
    }
    return x;
}

// the root of x without writing: the flatten pass must not shorten paths,
// since a path-halving store based on a stale read could overwrite a root
// that another warp has just stored (the unions before it may halve paths)
__device__ int db_root(const int* lab, int x)
{
    for (int n = 0; n < (1 << 24); ++n) {
        const int p = lab[x];
        if (p == x) return x;
        x = p;
    }
    return x;
}

__device__ void db_unite(int* lab, int a, int b)
{
    for (int n = 0; n < (1 << 24); ++n) {
        a = db_find(lab, a);
        b = db_find(lab, b);
        if (a == b) return;
        if (a < b) { const int t = a; a = b; b = t; }
        const int old = atomicMin(lab + a, b);
        if (old == a) return;
        a = old;
    }
}


// ------------------------------------------------------------------ teams ---
// t(), n(): the thread's index and the number of threads; sync(): a barrier
// that orders the team's memory; ctr: shared counters; tlev: shared level
// thresholds; sum(), max(): over the team, the same in every thread.  A
// cluster's barrier with the trips to L2 that follow it takes about 2.5 us, a
// CTA's well under one, so the parts with many short steps run in its first
// CTA alone: leads() and inner().
__device__ __forceinline__ long long warp_sum64(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

struct DbWarpShared {
    int ctr[4];
    float tlev[DB_MAX_LEVELS + 1];
};

// WIDE: a CTA or more, with the shared memory of one
struct WarpTeam {
    using Inner = WarpTeam;
    static constexpr bool CLUSTER = false, WIDE = false;
    __device__ bool leads() const { return true; }
    __device__ Inner inner() const { return *this; }
    int* ctr;
    float* tlev;
    __device__ WarpTeam(DbWarpShared& s) : ctr(s.ctr), tlev(s.tlev) {}
    __device__ int t() const { return threadIdx.x & 31; }
    __device__ int n() const { return 32; }
    __device__ void sync() const { __syncwarp(); }
    __device__ long long sum(long long v) const { return warp_sum64(v); }
    __device__ int max(int v) const { return __reduce_max_sync(0xffffffffu, v); }
};

struct DbGroupShared {
    int ctr[4];
    float tlev[DB_MAX_LEVELS + 1];
    long long part[DB_GW];
    int next;
};

// DB_GW warps of a CTA, on a named barrier of their own
struct GroupTeam {
    using Inner = GroupTeam;
    static constexpr bool CLUSTER = false, WIDE = false;
    DbGroupShared& s;
    int* ctr;
    float* tlev;
    __device__ GroupTeam(DbGroupShared& sh) : s(sh), ctr(sh.ctr), tlev(sh.tlev) {}
    __device__ bool leads() const { return true; }
    __device__ Inner inner() const { return *this; }
    __device__ int t() const { return threadIdx.x % (32 * DB_GW); }
    __device__ int n() const { return 32 * DB_GW; }
    __device__ void sync() const
    {
        asm volatile("barrier.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / (32 * DB_GW)), "n"(32 * DB_GW) : "memory");
    }
    template <class Op>
    __device__ long long all(long long v, Op op) const
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
        if ((threadIdx.x & 31) == 0) s.part[t() >> 5] = v;
        sync();
        v = s.part[0];
#pragma unroll
        for (int w = 1; w < DB_GW; ++w) v = op(v, s.part[w]);
        sync();
        return v;
    }
    __device__ long long sum(long long v) const { return all(v, [](long long a, long long b) { return a + b; }); }
    __device__ int max(int v) const { return (int)all(v, [](long long a, long long b) { return a > b ? a : b; }); }
};
static_assert(DB_NT % (32 * DB_GW) == 0 && DB_NT / (32 * DB_GW) < 16, "groups of whole warps, a named barrier each");

constexpr int DB_LIST = 1024;                // candidates of a round in shared memory; more go to global
struct DbCtaShared {
    int ctr[4];
    float tlev[DB_MAX_LEVELS + 1];
    long long part[DB_NT / 32], whole;
    int tree_i, tree_n, tree_odd;                          // where the tree stands
    int hist[DB_MAX_LEVELS], base[DB_MAX_LEVELS];          // growth: this CTA's pixels by level
    int total[DB_MAX_LEVELS], from[DB_MAX_LEVELS + 1];     // (first CTA) the team's; where each level's list starts
    __align__(16) int list[3][DB_LIST];                    // growth: the rounds' candidates
};
// growth: the box's pixels in the rest of the shared memory, two bytes of
// state each, when there are at most this many
constexpr int DB_BOX = 103000;
constexpr size_t DB_SMEM = 2 * (size_t)DB_BOX;

template <int CL>
struct CtaTeam {
    using Inner = CtaTeam<1>;
    static constexpr bool CLUSTER = CL > 1, WIDE = true;
    __device__ bool leads() const { return rank() == 0; }
    __device__ Inner inner() const { return Inner(s); }
    __device__ DbCtaShared& first() const
    {
        if constexpr (CL > 1) return *cg::this_cluster().map_shared_rank(&s, 0);
        else return s;
    }
    DbCtaShared& s;
    int* ctr;                  // the first CTA's
    float* tlev;               // each CTA its own copy
    __device__ CtaTeam(DbCtaShared& sh) : s(sh), ctr(sh.ctr), tlev(sh.tlev)
    {
        if constexpr (CL > 1) ctr = cg::this_cluster().map_shared_rank(sh.ctr, 0);
    }
    __device__ int rank() const { return CL > 1 ? (int)cg::this_cluster().block_rank() : 0; }
    __device__ int t() const { return rank() * DB_NT + threadIdx.x; }
    __device__ int n() const { return CL * DB_NT; }
    __device__ void sync() const
    {
        if constexpr (CL > 1) cg::this_cluster().sync();
        else __syncthreads();
    }
    template <class Op>
    __device__ long long all(long long v, Op op) const
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
        if ((threadIdx.x & 31) == 0) s.part[threadIdx.x >> 5] = v;
        __syncthreads();
        v = s.part[0];
        for (int w = 1; w < DB_NT / 32; ++w) v = op(v, s.part[w]);
        if constexpr (CL > 1) {
            if (threadIdx.x == 0) s.whole = v;
            sync();
            v = *cg::this_cluster().map_shared_rank(&s.whole, 0);
            for (int r = 1; r < CL; ++r) v = op(v, *cg::this_cluster().map_shared_rank(&s.whole, r));
        }
        sync();
        return v;
    }
    __device__ long long sum(long long v) const { return all(v, [](long long a, long long b) { return a + b; }); }
    __device__ int max(int v) const { return (int)all(v, [](long long a, long long b) { return a > b ? a : b; }); }
};

// a place in a list for each calling thread, one addition a warp
__device__ __forceinline__ int db_append(int* counter)
{
    const unsigned m = __activemask();
    const int lane = threadIdx.x & 31, lead = __ffs(m) - 1;
    int base = 0;
    if (lane == lead) base = atomicAdd(counter, __popc(m));
    return __shfl_sync(m, base, lead) + __popc(m & ((1u << lane) - 1u));
}

// atomicMin / atomicMax where the value at hand would change
__device__ __forceinline__ void db_min(int* p, int v)
{
    if (v < *(volatile int*)p) atomicMin(p, v);
}
__device__ __forceinline__ void db_max(int* p, int v)
{
    if (v > *(volatile int*)p) atomicMax(p, v);
}

// fs[rt] += mf, cnt[rt] += 1 for the lanes with rt >= 0 (the whole warp
// calls): most lanes share a few roots, whose sums go in one addition each;
// 64-bit sums by three 32-bit ones (exact modulo 2^64, as the additions are)
__device__ __forceinline__ void db_add(long long* fs, int* cnt, int rt, long long mf)
{
    const int lane = threadIdx.x & 31;
    unsigned todo = __ballot_sync(0xffffffffu, rt >= 0);
    for (int k = 0; k < 4 && todo; ++k) {
        const int lead = __ffs(todo) - 1;
        const int r0 = __shfl_sync(0xffffffffu, rt, lead);
        const bool mine = rt == r0;
        const unsigned long long u = mine ? (unsigned long long)mf : 0ull;
        const unsigned a = __reduce_add_sync(0xffffffffu, (unsigned)(u & 0xffffffu));
        const unsigned b = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 24 & 0xffffffu));
        const unsigned c = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 48));
        const unsigned grp = __ballot_sync(0xffffffffu, mine);
        if (lane == lead) {
            atomicAdd(reinterpret_cast<unsigned long long*>(fs + r0),
                      (unsigned long long)a + ((unsigned long long)b << 24) + ((unsigned long long)c << 48));
            atomicAdd(cnt + r0, __popc(grp));
        }
        todo &= ~grp;
    }
    if (todo >> lane & 1u) {
        atomicAdd(reinterpret_cast<unsigned long long*>(fs + rt), (unsigned long long)mf);
        atomicAdd(cnt + rt, 1);
    }
}

// --------------------------------------------------------- catalog rows ---
// sums over an object's pixels, coordinates about the box corner
struct DbSums {
    double sm, sx, sy, sxx, syy, sxy;
    long long c, ux, uy, uxx, uyy, uxy;
    float pk;                  // peak and its first pixel
    int pq, sat;
};
constexpr int DB_SUM_WORDS = 15;             // 8-byte words of a warp's partial sums

// over the warp's lanes: butterflies, so every lane has the same bits
__device__ __forceinline__ void db_warp_sums(DbSums& o)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        auto dd = [&](double& v) { v += __shfl_xor_sync(0xffffffffu, v, d); };
        auto ll = [&](long long& v) { v += __shfl_xor_sync(0xffffffffu, v, d); };
        dd(o.sm); dd(o.sx); dd(o.sy); dd(o.sxx); dd(o.syy); dd(o.sxy);
        ll(o.c); ll(o.ux); ll(o.uy); ll(o.uxx); ll(o.uyy); ll(o.uxy);
        const float pk = __shfl_xor_sync(0xffffffffu, o.pk, d);
        const int pq = __shfl_xor_sync(0xffffffffu, o.pq, d);
        if (pk > o.pk || (pk == o.pk && pq < o.pq)) { o.pk = pk; o.pq = pq; }
        o.sat |= __shfl_xor_sync(0xffffffffu, o.sat, d);
    }
}

template <bool F32>
__device__ __forceinline__ DbSums db_object_sums(const Image& im, const DbScratch& s, const int* cur, int k, int x0, int y0,
                                                 int w, int wh, int hx, int hy, int bx0, int by0, int bw, int area, int t,
                                                 int n)
{
    DbSums o = {};
    o.pk = -INFINITY;
    o.pq = INT_MAX;
    for (int i = t; i < area; i += n) {
        const int qy = by0 + i / bw, qx = bx0 + i % bw, q = qy * w + qx;
        if (cur[q] != k) continue;
        const float mv = s.mh[(qy + hy) * wh + qx + hx];
        const double m = (double)mv, xm = qx * m, ym = qy * m;    // products exact in float64
        o.sm += m; o.sx += xm; o.sy += ym;
        o.sxx += qx * xm; o.syy += qy * ym; o.sxy += qy * xm;
        o.c += 1; o.ux += qx; o.uy += qy;
        o.uxx += (long long)qx * qx; o.uyy += (long long)qy * qy; o.uxy += (long long)qx * qy;
        if (mv > o.pk || (mv == o.pk && q < o.pq)) { o.pk = mv; o.pq = q; }
        if (im.sat > 0.f) {
            bool bad;
            if (load_px<F32>(im, x0 + qx, y0 + qy, bad) >= im.sat) o.sat = 1;
        }
    }
    db_warp_sums(o);
    return o;
}

__device__ __forceinline__ void db_emit(const DeblendArgs& A, const DbSums& v, uint32_t L, uint32_t label, int x0, int y0,
                                        int w, int bx0, int bx1, int by0, int by1)
{
    const int idx = atomicAdd(A.obj_count, 1);
    if (idx >= A.obj_stage_cap) {
        set_status(A.status, GP_ERR_CAPACITY);
        return;
    }
    DbObj o;
    o.label = label;
    o.parent = L;
    o.npix = (int)v.c;
    uint32_t fl = v.sat ? GP_FLAG_SAT : 0u;
    double xm, ym, x2, y2, xy;
    if (v.sm > 0.0) {
        xm = v.sx / v.sm; ym = v.sy / v.sm;
        x2 = v.sxx / v.sm - xm * xm; y2 = v.syy / v.sm - ym * ym; xy = v.sxy / v.sm - xm * ym;
    } else {
        const double c = (double)v.c;
        xm = (double)v.ux / c; ym = (double)v.uy / c;
        x2 = (double)v.uxx / c - xm * xm; y2 = (double)v.uyy / c - ym * ym; xy = (double)v.uxy / c - xm * ym;
        fl |= GP_FLAG_CENTROID_FALLBACK;
    }
    o.flux = v.sm;
    o.x = xm + x0; o.y = ym + y0; o.x2 = x2; o.y2 = y2; o.xy = xy;
    o.xmin = x0 + bx0; o.xmax = x0 + bx1; o.ymin = y0 + by0; o.ymax = y0 + by1;
    o.peak = v.pk;
    o.xpeak = x0 + v.pq % w; o.ypeak = y0 + v.pq / w;
    o.flags = fl;
    A.obj[idx] = o;
}

// ------------------------------------------------------------ a segment ---
// active pixels that one CTA of a cluster works on alone (crowded 17 MP field,
// 512, 2,048 and 8,192: 1.91, 1.91 and 1.97 ms)
constexpr int DB_TREE_ONE = 2048;

// the branch tree from level i on, over the list lst of the nl pixels still
// active, down to a list of `least`
template <class Team>
__device__ __forceinline__ void db_tree(const DeblendArgs& A, const Team T, const DbScratch& s, int w, int Ar, double cthr,
                                        int least, int& i, int& nl, int*& lst, int*& lnx)
{
    const int t = T.t(), n = T.n();
    for (; i + 1 < A.nthresh && nl > least; ++i) {
        const float tl = T.tlev[i + 1];
        for (int k = t; k < nl; k += n) {
            const int q = lst[k];
            s.lab[q] = s.nu[q] > tl ? q : -1;
            s.fs[q] = 0; s.cnt[q] = 0; s.sig[q] = 0;
        }
        if (t == 0) { s.fs[Ar] = 0; s.cnt[Ar] = 0; s.sig[Ar] = 0; T.ctr[1 + (i & 1)] = 0; }
        T.sync();
        for (int k = t; k < nl; k += n) {
            const int q = lst[k];
            if (s.lab[q] < 0) continue;
            const int qy = q / w, qx = q - qy * w;
            // the neighbours before q in raster order; N touches the others,
            // W touches NW, so those unite among themselves
            const bool hw = qx > 0 && s.lab[q - 1] >= 0;
            const int u = q - w;
            if (qy > 0 && s.lab[u] >= 0) {
                db_unite(s.lab, q, u);
            } else {
                if (hw) db_unite(s.lab, q, q - 1);
                else if (qy > 0 && qx > 0 && s.lab[u - 1] >= 0) db_unite(s.lab, q, u - 1);
                if (qy > 0 && qx + 1 < w && s.lab[u + 1] >= 0) db_unite(s.lab, q, u + 1);
            }
        }
        T.sync();
        // roots into a second array (own2 is free until the growth), and their sums
        int* root = s.own2;
        for (int k0 = t - (threadIdx.x & 31); k0 < nl; k0 += n) {
            const int k = k0 + (threadIdx.x & 31);
            int rt = -1;
            long long mf = 0;
            if (k < nl) {
                const int q = lst[k];
                if (s.lab[q] >= 0) {
                    rt = db_root(s.lab, q);
                    mf = s.mf[q];
                }
                root[q] = rt;
            }
            db_add(s.fs, s.cnt, rt, mf);
        }
        T.sync();
        // a significant branch marks its parent node (the active node of its pixels)
        for (int k = t; k < nl; k += n) {
            const int q = lst[k];
            if (root[q] != q) continue;
            if (s.cnt[q] >= A.minarea && (double)s.fs[q] > cthr) {
                atomicOr(s.sig + q, 1);
                atomicOr(s.sig + s.act[q], 2);
            }
        }
        T.sync();
        for (int k = t; k < nl; k += n) {
            const int q = lst[k];
            const int node = s.act[q];
            if (!(s.sig[node] & 2)) {           // no significant child: the node is a seed
                s.seed[q] = node + 1;
                s.act[q] = -1;
                s.lab[q] = -1;
            } else if (root[q] >= 0 && (s.sig[root[q]] & 1)) {
                s.act[q] = root[q];
                lnx[db_append(&T.ctr[1 + (i & 1)])] = q;
            } else {
                s.act[q] = -1;
                s.lab[q] = -1;
            }
        }
        T.sync();
        int* tmp = lst; lst = lnx; lnx = tmp;
        nl = T.ctr[1 + (i & 1)];
    }
}

// The rounds on a box in shared memory.  A pixel's state, 16 bits of a word
// that it shares with a neighbour: 0 unassigned, ST_CAND a candidate, else its
// rank, with ST_ODD or ST_EVEN added in the round it was assigned in (by the
// round's parity) and taken off in the next: in a round, ranks are read from
// pixels without that round's mark.  Within a round an unassigned pixel can
// only become a candidate, so setting ST_CAND's bits claims it.
// While the rounds run, threads change and read the two states of a word at
// once, so every change is an atomic of the word and every read a volatile
// load of it: no access meets one of another size.
constexpr unsigned ST_ODD = 0x4000u, ST_EVEN = 0x8000u, ST_CAND = 0xc000u, ST_RANK = 0x3fffu;

__device__ __forceinline__ void db_rounds_shared(const DeblendArgs& A, DbCtaShared& S, const DbScratch& s, int w, int h,
                                                 unsigned short* state)
{
    const int t = threadIdx.x, n = DB_NT;
    // lists of up to DB_LIST pixels in shared memory, the rest in lab, act and seed
    int* const more[3] = {s.lab, s.act, s.seed};
    auto get = [&](int l, int k) { return k < DB_LIST ? S.list[l][k] : more[l][k]; };
    auto put = [&](int l, int k, int q) {
        if (k < DB_LIST) S.list[l][k] = q;
        else more[l][k] = q;
    };
    auto neighbours = [&](int q, int (&o)[8]) {
        const int qy = q / w, qx = q - qy * w;
        const bool l = qx > 0, r = qx + 1 < w, u = qy > 0, d = qy + 1 < h;
        o[0] = u && l ? -w - 1 : 0; o[1] = u ? -w : 0; o[2] = u && r ? -w + 1 : 0; o[3] = l ? -1 : 0;
        o[4] = r ? 1 : 0; o[5] = d && l ? w - 1 : 0; o[6] = d ? w : 0; o[7] = d && r ? w + 1 : 0;
    };
    unsigned* const words = reinterpret_cast<unsigned*>(state);
    auto at = [](int q) { return 16 * (q & 1); };
    auto load = [&](int q) { return *(const volatile unsigned*)(words + (q >> 1)) >> at(q) & 0xffffu; };
    int c = 0, round = 0, last = 0;          // last: pixels assigned in the round before, in list c - 1
    for (int i = A.nthresh - 1; i >= 0; --i) {
        const float tl = i > 0 ? S.tlev[i] : -INFINITY;    // nu > -inf: any pixel of the segment
        for (int k = S.from[i] + t; k < S.from[i + 1]; k += n) {
            const int q = s.first[k];
            int o[8];
            neighbours(q, o);
            bool any = false;
#pragma unroll
            for (int j = 0; j < 8; ++j) any = any || (o[j] && (load(q + o[j]) & ST_RANK) != 0);
            if (any) {
                atomicOr(words + (q >> 1), ST_CAND << at(q));
                put(c, db_append(&S.ctr[c]), q);
            }
        }
        __syncthreads();
        for (;;) {
            const int nc = S.ctr[c], cn = c == 2 ? 0 : c + 1, cp = cn == 2 ? 0 : cn + 1;   // cp: the round before's
            if (nc == 0 && last == 0) break;
            ++round;
            const unsigned now = round & 1 ? ST_ODD : ST_EVEN;
            if (t == 0) S.ctr[cp] = 0;       // (its length is in `last`; filled again in the next round)
            for (int k = t; k < last; k += n) {
                const int q = get(cp, k);
                atomicAnd(words + (q >> 1), ~(ST_CAND << at(q)));
            }
            for (int k = t; k < nc; k += n) {
                const int q = get(c, k);
                int o[8];
                unsigned st[8], best = ST_CAND;
                neighbours(q, o);
#pragma unroll
                for (int j = 0; j < 8; ++j) st[j] = o[j] ? load(q + o[j]) : ST_CAND;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (st[j] != 0 && (st[j] & ST_CAND) != ST_CAND && !(st[j] & now)) best = min(best, st[j] & ST_RANK);
                atomicXor(words + (q >> 1), (ST_CAND ^ (best | now)) << at(q));     // from ST_CAND
                // claim the unassigned neighbours in the level set
                float nu[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) nu[j] = st[j] == 0 ? s.nu[q + o[j]] : -INFINITY;
                unsigned old[8], won = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int p = q + o[j], sh = at(p);
                    old[j] = nu[j] > tl ? atomicOr(words + (p >> 1), ST_CAND << sh) >> sh & 0xffffu : 1u;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) won |= old[j] == 0u ? 1u << j : 0u;
                if (won) {
                    int k2 = atomicAdd(&S.ctr[cn], __popc(won));
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (won >> j & 1u) put(cn, k2++, q + o[j]);
                }
            }
            __syncthreads();
            last = nc;
            c = cn;
        }
        __syncthreads();                     // every thread has seen the counter at zero before it counts again
    }
}

// Growth within the level sets, from the highest level down, in synchronous
// rounds: in a round every unassigned pixel of the level set with an assigned
// 8-neighbour takes the smallest object rank among the neighbours assigned
// before the round.  A level's first round looks at the pixels that are new at
// it (one of a higher level beside an assigned pixel would have been assigned
// there): the larger teams list the pixels by level first, a warp scans its
// small box.  After that a pixel can become a candidate only through a
// neighbour assigned in the round before, so each later round visits the
// neighbours of the last round's pixels.  Within a round a candidate may be
// given its rank and its unassigned neighbours listed for the next one at
// once: ranks are read from pixels stamped before the round only.
// Rounds are many (some 250) and short (a hundred pixels): one CTA of a
// cluster makes them, on a copy of the box in its shared memory where that
// fits (db_rounds_shared), else in global memory with the eight neighbours'
// loads together.  A round took 5.5 us with the cluster's barrier and one
// load after the other, 2.5 in one CTA; in shared memory about 1.
// own: the object rank of each pixel (0 none); own2: the round in which it was
// assigned (seeds 0; -1 unassigned, -2 a candidate of the coming round); lists:
// lab and act in turn, their lengths in three counters in turn (read, filled,
// cleared), zero on entry; first: the pixels by level.
template <class Team>
__device__ __forceinline__ void db_growth(const DeblendArgs& A, const Team T, const DbScratch& s, int w, int h, int Ar)
{
    extern __shared__ __align__(16) unsigned char box[];
    constexpr bool BUCKETS = Team::WIDE;
    int* cur = s.own;
    int* stamp = s.own2;
    if constexpr (BUCKETS) {
        auto level_of = [&](float nu) {          // the largest i with nu > tlev[i], or 0
            int lo = 0, hi = A.nthresh;
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (nu > T.tlev[mid]) lo = mid;
                else hi = mid;
            }
            return lo;
        };
        DbCtaShared& own = T.s;
        DbCtaShared& all = T.first();
        if (threadIdx.x < DB_MAX_LEVELS) own.hist[threadIdx.x] = own.total[threadIdx.x] = 0;
        T.sync();
        for (int q = T.t(); q < Ar; q += T.n())
            if (cur[q] == 0 && s.nu[q] > -INFINITY) atomicAdd(&own.hist[level_of(s.nu[q])], 1);
        __syncthreads();
        if (threadIdx.x < DB_MAX_LEVELS) {
            own.base[threadIdx.x] = atomicAdd(&all.total[threadIdx.x], own.hist[threadIdx.x]);
            own.hist[threadIdx.x] = 0;
        }
        T.sync();
        if (threadIdx.x < DB_MAX_LEVELS) own.from[threadIdx.x + 1] = all.total[threadIdx.x];
        __syncthreads();
        if (threadIdx.x == 0) {
            own.from[0] = 0;
            for (int i = 1; i <= DB_MAX_LEVELS; ++i) own.from[i] += own.from[i - 1];
        }
        __syncthreads();
        for (int q = T.t(); q < Ar; q += T.n())
            if (cur[q] == 0 && s.nu[q] > -INFINITY) {
                const int i = level_of(s.nu[q]);
                s.first[own.from[i] + own.base[i] + atomicAdd(&own.hist[i], 1)] = q;
            }
        T.sync();
        if (!T.leads()) return;
        if (Ar <= DB_BOX) {
            unsigned short* state = reinterpret_cast<unsigned short*>(box);
            for (int q = threadIdx.x; q < Ar; q += DB_NT) state[q] = (unsigned short)cur[q];
            __syncthreads();
            db_rounds_shared(A, own, s, w, h, state);
            for (int q = threadIdx.x; q < Ar; q += DB_NT) cur[q] = state[q];
            return;
        }
    }
    const typename Team::Inner I = T.inner();
    const int t = I.t(), n = I.n();
    int* lc = s.lab;
    int* ln = s.act;
    int round = 0, c = 0;
    for (int i = A.nthresh - 1; i >= 0; --i) {
        const float tl = I.tlev[i];
        auto eligible = [&](float nu) { return nu > -INFINITY && (i == 0 || nu > tl); };
        // offsets of the neighbours of q inside the box (0: outside)
        auto neighbours = [&](int q, int (&o)[8]) {
            const int qy = q / w, qx = q - qy * w;
            const bool l = qx > 0, r = qx + 1 < w, u = qy > 0, d = qy + 1 < h;
            o[0] = u && l ? -w - 1 : 0; o[1] = u ? -w : 0; o[2] = u && r ? -w + 1 : 0; o[3] = l ? -1 : 0;
            o[4] = r ? 1 : 0; o[5] = d && l ? w - 1 : 0; o[6] = d ? w : 0; o[7] = d && r ? w + 1 : 0;
        };
        auto first_round = [&](int q) {
            int o[8], v[8];
            neighbours(q, o);
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = o[j] ? cur[q + o[j]] : 0;
            int any = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) any |= v[j];
            if (any > 0) {
                stamp[q] = -2;
                lc[db_append(&I.ctr[c])] = q;
            }
        };
        // the counter c is zero here
        if constexpr (BUCKETS) {
            const int k1 = T.s.from[i + 1];
            for (int k = T.s.from[i] + t; k < k1; k += n) first_round(s.first[k]);
        } else {
            for (int q = t; q < Ar; q += n)
                if (cur[q] == 0 && eligible(s.nu[q])) first_round(q);
        }
        I.sync();
        for (;;) {
            const int nc = I.ctr[c], cn = c == 2 ? 0 : c + 1, cz = cn == 2 ? 0 : cn + 1;
            if (nc == 0) break;
            ++round;
            if (t == 0) I.ctr[cz] = 0;
            for (int k = t; k < nc; k += n) {
                const int q = lc[k];
                int o[8], st[8], v[8];
                float nu[8];
                neighbours(q, o);
#pragma unroll
                for (int j = 0; j < 8; ++j) st[j] = o[j] ? stamp[q + o[j]] : -3;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    v[j] = st[j] >= 0 && st[j] < round ? cur[q + o[j]] : INT_MAX;
                    nu[j] = st[j] == -1 ? s.nu[q + o[j]] : -INFINITY;
                }
                int best = INT_MAX;
#pragma unroll
                for (int j = 0; j < 8; ++j) best = min(best, v[j]);
                cur[q] = best;
                stamp[q] = round;
                int old[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) old[j] = eligible(nu[j]) ? atomicCAS(stamp + q + o[j], -1, -2) : 0;
                int won = 0;
#pragma unroll
                for (int j = 0; j < 8; ++j) won += old[j] == -1;
                if (won) {
                    int k2 = atomicAdd(&I.ctr[cn], won);
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (old[j] == -1) ln[k2++] = q + o[j];
                }
            }
            I.sync();
            int* tmp = lc; lc = ln; ln = tmp;
            c = cn;
        }
        // every thread has read the counter c (zero) before the next level's
        // candidates are counted in it
        I.sync();
    }
}

template <bool F32, class Team>
__device__ __noinline__ void db_segment(const DeblendArgs& A, int ci, const Team T)
{
    const int t = T.t(), n = T.n();
    const Image& im = A.im;
    const int W = im.W, H = im.H;
    const int hx = A.kw / 2, hy = A.kh / 2;
    if (A.off[ci] < 0) return;                         // no room: left as it is (status set)
    const int rc = A.cand[ci], r = rc < 0 ? ~rc : rc;
    const uint32_t L = A.label[r];
    const int x0 = A.xmin[r], x1 = A.xmax[r], y0 = A.ymin[r], y1 = A.ymax[r];
    const int w = x1 - x0 + 1, h = y1 - y0 + 1, Ar = w * h;
    const int wh = w + 2 * hx, hh = h + 2 * hy, AH = wh * hh;
    DbScratch s = db_scratch(A.scratch + A.off[ci], Ar, AH);
    // ---- m over the box and halo, then nu and fixed-point m in the segment
    for (int q = t; q < AH; q += n) {
        const int qy = q / wh, qx = q - qy * wh;
        int x = x0 - hx + qx, y = y0 - hy + qy;
        if ((unsigned)x >= (unsigned)W) x = mirror_idx(x, W);
        if ((unsigned)y >= (unsigned)H) y = mirror_idx(y, H);
        bool bad;
        const float v = load_px<F32>(im, x, y, bad);
        s.mh[q] = bad ? 0.f : v - spline_eval(A.sb, (float)x, (float)y);
    }
    if (t == 0) T.ctr[0] = T.ctr[1] = T.ctr[2] = T.ctr[3] = 0;
    T.sync();
    long long tot = 0;
    float numax = -INFINITY;
    for (int q = t; q < Ar; q += n) {
        const int qy = q / w, qx = q - qy * w;
        const int x = x0 + qx, y = y0 + qy;
        const bool in = A.seg[(int64_t)y * W + x] == L;
        float nu = -1.f;
        long long mf = 0;
        if (in) {
            float F = 0.f;
            for (int v = 0; v < A.kh; ++v)
                for (int u = 0; u < A.kw; ++u) F = fmaf(A.taps[v * A.kw + u], s.mh[(qy + v) * wh + qx + u], F);
            const float sg = spline_eval(A.sr, (float)x, (float)y);
            nu = sg > 0.f ? F / sg : 0.f;
            mf = llrint((double)s.mh[(qy + hy) * wh + qx + hx] * DB_FIX);
            numax = fmaxf(numax, nu);
        }
        s.nu[q] = in ? nu : -INFINITY;
        s.mf[q] = mf;
        tot += mf;
        s.act[q] = in ? Ar : -1;              // level 0: the whole segment is node Ar
        s.seed[q] = 0;
    }
    // floats in the order of ints
    const int nk = __float_as_int(numax + 0.f);
    const long long total = T.sum(tot);
    const int mk = T.max(nk < 0 ? nk ^ 0x7fffffff : nk);
    const float numax_all = __int_as_float(mk < 0 ? mk ^ 0x7fffffff : mk);
    if (!(total > 0) || !(numax_all > A.thresh)) return;
    T.sync();
    // a branch always holds a local maximum of nu (its largest value), so a
    // segment with fewer than two (plateaus counted per pixel) cannot split
    int nmax = 0;
    for (int q = t; q < Ar; q += n) {
        const float v = s.nu[q];
        if (v == -INFINITY) continue;
        const int qy = q / w, qx = q - qy * w;
        bool mx = true;
        for (int dy = -1; dy <= 1 && mx; ++dy)
            for (int dx = -1; dx <= 1; ++dx) {
                const int yy = qy + dy, xx = qx + dx;
                if ((dy || dx) && yy >= 0 && yy < h && xx >= 0 && xx < w && s.nu[yy * w + xx] > v) { mx = false; break; }
            }
        nmax += mx ? 1 : 0;
    }
    if (T.sum(nmax) < 2) return;
    const double cthr = A.mincont * (double)total;
    const double lr = log((double)numax_all / (double)A.thresh);
    // t_i = thresh (nu_max / thresh)^(i / nthresh), once per level, in
    // float64, rounded down to float: for a float nu, nu > t_i exactly
    // when nu > rd(t_i), so every comparison below is one of floats
    for (int i = t % DB_NT; i <= A.nthresh; i += n < DB_NT ? n : DB_NT)
        T.tlev[i] = __double2float_rd((double)A.thresh * exp(lr * (double)i / (double)A.nthresh));
    // ---- the branch tree, one level at a time, over the list of the
    // pixels still active (own: this level's list, first: the next
    // level's).  A pixel leaves the list when it leaves the tree, and its
    // lab is then -1 for good; the nodes the listed pixels point to are
    // listed pixels themselves (a significant branch's root stays in it)
    // or node Ar.  Roots are the components' smallest pixels and the
    // sums are exact, so the list order does not matter.
    int* lst = s.own;
    int* lnx = s.first;
    for (int q = t; q < Ar; q += n) {
        s.lab[q] = -1;
        if (s.act[q] >= 0) lst[db_append(&T.ctr[0])] = q;
    }
    T.sync();
    int nl = T.ctr[0];
    int level = 0;
    if constexpr (Team::CLUSTER) {
        // the whole cluster while the list is long, then its first CTA
        db_tree(A, T, s, w, Ar, cthr, DB_TREE_ONE, level, nl, lst, lnx);
        T.sync();                    // every thread has read the list's length
        if (T.leads()) {
            db_tree(A, T.inner(), s, w, Ar, cthr, 0, level, nl, lst, lnx);
            if (t == 0) { T.s.tree_n = nl; T.s.tree_odd = lst == s.first; }
        }
        T.sync();
        nl = T.first().tree_n;
        lst = T.first().tree_odd ? s.first : s.own;
    } else {
        db_tree(A, T, s, w, Ar, cthr, 0, level, nl, lst, lnx);
    }
    for (int k = t; k < nl; k += n) {
        const int q = lst[k];
        s.seed[q] = s.act[q] + 1;
    }
    T.sync();
    // ---- the seeds, in the order of their first pixels (fs is free: seeds
    // and their ids)
    int* seeds = reinterpret_cast<int*>(s.fs);
    int* seedid = seeds + Ar + 1;
    for (int q = t; q <= Ar; q += n) s.first[q] = INT_MAX;
    if (t == 0) T.ctr[0] = 0;
    T.sync();
    for (int q = t; q < Ar; q += n)
        if (s.seed[q]) db_min(s.first + s.seed[q] - 1, q);
    T.sync();
    for (int q = t; q < Ar; q += n) {
        if (s.seed[q] && s.first[s.seed[q] - 1] == q) {
            const int k = db_append(&T.ctr[0]);
            if (k < DB_MAX_SEEDS) { seeds[k] = q; seedid[k] = s.seed[q] - 1; }
        }
    }
    T.sync();
    const int ns = T.ctr[0];
    if (ns > DB_MAX_SEEDS) {
        if (t == 0) set_status(A.status, GP_ERR_CAPACITY);
        return;
    }
    if (ns < 2) return;
    // rank of each seed by its first pixel (first pixels are distinct)
    for (int k = t; k < ns; k += n) {
        int rk = 0;
        for (int j = 0; j < ns; ++j) rk += seeds[j] < seeds[k];
        s.cnt[seedid[k]] = rk + 1;
    }
    T.sync();
    // own: the object rank of each pixel (0 none); own2: the round in which
    // the pixel was assigned (seeds 0; -1 unassigned, -2 a candidate of
    // the coming round)
    for (int q = t; q < Ar; q += n) {
        const int v = s.seed[q] ? s.cnt[s.seed[q] - 1] : 0;
        s.own[q] = v;
        s.own2[q] = v > 0 ? 0 : -1;
    }
    if (t == 0) T.ctr[0] = T.ctr[1] = T.ctr[2] = 0;
    T.sync();
    // ---- the other pixels
    int* cur = s.own;
    db_growth(A, T, s, w, h, Ar);
    T.sync();
    // ---- each object's box and first pixel, its label, its pixels' labels
    // (lab, act, seed and cnt are free: the boxes; sig: the first pixels)
    int* bx0 = s.lab;
    int* bx1 = s.act;
    int* by0 = s.seed;
    int* by1 = s.cnt;
    int* fp = s.sig;
    for (int k = t; k < ns; k += n) {
        bx0[k] = by0[k] = fp[k] = INT_MAX;
        bx1[k] = by1[k] = -1;
    }
    T.sync();
    for (int q = t; q < Ar; q += n) {
        const int o = cur[q] - 1;
        if (o < 0) continue;
        const int qy = q / w, qx = q - qy * w;
        db_min(fp + o, q);
        db_min(bx0 + o, qx); db_max(bx1 + o, qx);
        db_min(by0 + o, qy); db_max(by1 + o, qy);
    }
    T.sync();
    auto label = [&](int k) { return (uint32_t)((y0 + fp[k] / w) * W + x0 + fp[k] % w) + 1u; };
    for (int q = t; q < Ar; q += n) {
        const int o = cur[q] - 1;
        if (o >= 0) A.seg[(int64_t)(y0 + q / w) * W + x0 + q % w] = label(o);
    }
    // ---- each object's catalog row: a warp for each, a CTA for those with a
    // large box, whose warps' sums the first warp adds
    const int lane = threadIdx.x & 31, gw = t >> 5, nw = n >> 5;
    for (int k = gw; k < ns; k += nw) {
        const int bw = bx1[k] - bx0[k] + 1, area = bw * (by1[k] - by0[k] + 1);
        if (Team::WIDE && area > DB_ROW) continue;
        const DbSums v = db_object_sums<F32>(im, s, cur, k + 1, x0, y0, w, wh, hx, hy, bx0[k], by0[k], bw, area, lane, 32);
        if (lane == 0) db_emit(A, v, L, label(k), x0, y0, w, bx0[k], bx1[k], by0[k], by1[k]);
    }
    if constexpr (Team::WIDE) {
        static_assert(sizeof(T.s.list) >= sizeof(long long) * DB_SUM_WORDS * (DB_NT / 32), "the warps' sums fit");
        long long* part = reinterpret_cast<long long*>(T.s.list);
        int large = 0;
        for (int k = 0; k < ns; ++k) {
            const int bw = bx1[k] - bx0[k] + 1, area = bw * (by1[k] - by0[k] + 1);
            if (area <= DB_ROW || large++ % (n / DB_NT) != t / DB_NT) continue;
            DbSums v = db_object_sums<F32>(im, s, cur, k + 1, x0, y0, w, wh, hx, hy, bx0[k], by0[k], bw, area,
                                           threadIdx.x, DB_NT);
            if (lane == 0) {
                long long* p = part + (threadIdx.x >> 5) * DB_SUM_WORDS;
                const double d[6] = {v.sm, v.sx, v.sy, v.sxx, v.syy, v.sxy};
                for (int j = 0; j < 6; ++j) p[j] = __double_as_longlong(d[j]);
                p[6] = v.c; p[7] = v.ux; p[8] = v.uy; p[9] = v.uxx; p[10] = v.uyy; p[11] = v.uxy;
                p[12] = __float_as_int(v.pk); p[13] = v.pq; p[14] = v.sat;
            }
            __syncthreads();
            if (threadIdx.x < 32) {
                static_assert(DB_NT / 32 == 32, "a warp's sums a lane");
                const long long* p = part + lane * DB_SUM_WORDS;
                v.sm = __longlong_as_double(p[0]); v.sx = __longlong_as_double(p[1]); v.sy = __longlong_as_double(p[2]);
                v.sxx = __longlong_as_double(p[3]); v.syy = __longlong_as_double(p[4]); v.sxy = __longlong_as_double(p[5]);
                v.c = p[6]; v.ux = p[7]; v.uy = p[8]; v.uxx = p[9]; v.uyy = p[10]; v.uxy = p[11];
                v.pk = __int_as_float((int)p[12]); v.pq = (int)p[13]; v.sat = (int)p[14];
                db_warp_sums(v);
                if (lane == 0) db_emit(A, v, L, label(k), x0, y0, w, bx0[k], bx1[k], by0[k], by1[k]);
            }
            __syncthreads();
        }
    }
    if (t == 0) {
        atomicAdd(A.counts, 1);
        atomicAdd(A.counts + 1, ns);
    }
}

template <bool F32>
__global__ void __cluster_dims__(DB_CL, 1, 1) __launch_bounds__(DB_NT, 1) k_deblend(const __grid_constant__ DeblendArgs A)
{
    const int nbig = min(A.ctl[DBC_BIG], DB_MAX_BIG), nmid = A.ctl[DBC_N], nsmall = A.ctl[DBC_SMALL];
    __shared__ DbCtaShared sh;
    __shared__ DbGroupShared gs[DB_NT / (32 * DB_GW)];
    __shared__ DbWarpShared ws[DB_NT / 32];
    __shared__ int next;
    // the next candidate of the front that is (not) a group's
    auto claim = [&](int* counter, bool group) {
        int c;
        do c = atomicAdd(counter, 1);
        while (c < nmid && (A.cand[c] < 0) != group);
        return c;
    };
    {
        const CtaTeam<DB_CL> T(sh);
        const auto cl = cg::this_cluster();
        int* const nx = cl.map_shared_rank(&next, 0);
        for (;;) {
            if (T.t() == 0) next = atomicAdd(A.ctl + DBC_NEXT_BIG, 1);
            T.sync();
            const int b = *nx;
            T.sync();
            if (b >= nbig) break;
            db_segment<F32>(A, A.ctl[DBC_LIST + b], T);
        }
    }
    for (;;) {
        const CtaTeam<1> T(sh);
        __syncthreads();
        if (threadIdx.x == 0) next = claim(A.ctl + DBC_NEXT, false);
        __syncthreads();
        const int c = next;
        if (c >= nmid) break;
        bool big = false;
        for (int b = 0; b < nbig; ++b) big = big || A.ctl[DBC_LIST + b] == c;
        if (!big) db_segment<F32>(A, c, T);
    }
    {
        DbGroupShared& g = gs[threadIdx.x / (32 * DB_GW)];
        const GroupTeam T(g);
        for (;;) {
            T.sync();
            if (T.t() == 0) g.next = claim(A.ctl + DBC_NEXT_MED, true);
            T.sync();
            const int c = g.next;
            if (c >= nmid) break;
            db_segment<F32>(A, c, T);
        }
    }
    const WarpTeam T(ws[threadIdx.x >> 5]);
    for (;;) {
        int c = 0;
        if ((threadIdx.x & 31) == 0) c = atomicAdd(A.ctl + DBC_NEXT_SMALL, 1);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= nsmall) break;
        db_segment<F32>(A, A.cap - 1 - c, T);
        __syncwarp();
    }
}

// candidates: rows with at least 2 minarea pixels, their scratch bytes; the
// larger ones from the front of the arrays (a group's as ~row), the small ones
// from the back
__global__ void __launch_bounds__(256) k_db_select(const int* __restrict__ n_dev, int cap,
                                                   const int* __restrict__ npix, const int* __restrict__ xmin,
                                                   const int* __restrict__ xmax, const int* __restrict__ ymin,
                                                   const int* __restrict__ ymax, int minarea, int hx, int hy,
                                                   int* cand, int* ctl, int64_t* bytes)
{
    const int n = min(*n_dev, cap);
    const int warps_most = n > DB_MANY ? DB_SMALL_MANY : DB_SMALL;
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
        if (npix[r] < 2 * minarea) continue;
        const int64_t w = xmax[r] - xmin[r] + 1, h = ymax[r] - ymin[r] + 1;
        const bool small = w * h <= warps_most;
        const int i = atomicAdd(ctl + (small ? DBC_SMALL : DBC_N), 1);
        const int k = small ? cap - 1 - i : i;
        if (w * h > DB_BIG) {
            const int b = atomicAdd(ctl + DBC_BIG, 1);
            if (b < DB_MAX_BIG) ctl[DBC_LIST + b] = k;
        }
        cand[k] = !small && w * h <= DB_MED ? ~r : r;
        bytes[k] = db_scratch_bytes(w * h, (w + 2 * hx) * (h + 2 * hy));
    }
}

// scratch offsets (exclusive scan of the bytes, one CTA); a candidate beyond
// the scratch gets -1 and the status records it
__global__ void __launch_bounds__(1024) k_db_offsets(const int* __restrict__ ctl, int cap, int64_t* bytes_off,
                                                     int64_t cap_bytes, int* status)
{
    __shared__ long long part[32];
    __shared__ long long carry;
    const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
    const int nlarge = ctl[DBC_N], n = nlarge + ctl[DBC_SMALL];
    if (t == 0) carry = 0;
    __syncthreads();
    for (int c0 = 0; c0 < n; c0 += 1024) {
        const bool in = c0 + t < n;
        const int i = c0 + t < nlarge ? c0 + t : cap - 1 - (c0 + t - nlarge);
        const long long v = in ? bytes_off[i] : 0;
        long long inc = v;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) part[wp] = inc;
        __syncthreads();
        if (wp == 0) {
            long long p = part[lane];
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, p, o);
                if (lane >= o) p += y;
            }
            part[lane] = p;
        }
        __syncthreads();
        const long long base = carry + (wp ? part[wp - 1] : 0);
        if (in) {
            const long long o = base + inc - v;
            const bool fits = o + v <= cap_bytes;
            bytes_off[i] = fits ? o : -1;
            if (!fits) set_status(status, GP_ERR_CAPACITY);
        }
        __syncthreads();
        if (t == 1023) carry = base + inc;
        __syncthreads();
    }
}

// the staged object rows in label order (rank by count; labels are distinct),
// the labels read by tiles through shared memory
__global__ void __launch_bounds__(256) k_db_place(const DbObj* __restrict__ obj, const int* __restrict__ obj_count,
                                                  int stage_cap, gp_catalog out)
{
    __shared__ uint32_t lab[1024];
    const int n = min(*obj_count, stage_cap);
    for (int i0 = blockIdx.x * blockDim.x; i0 < n; i0 += gridDim.x * blockDim.x) {
        const int i = i0 + threadIdx.x;
        const uint32_t L = i < n ? obj[i].label : 0u;
        int rk = 0;
        for (int j0 = 0; j0 < n; j0 += 1024) {
            const int m = min(1024, n - j0);
            __syncthreads();
            for (int j = threadIdx.x; j < m; j += 256) lab[j] = obj[j0 + j].label;
            __syncthreads();
            for (int j = 0; j < m; ++j) rk += lab[j] < L;
        }
        if (i >= n || rk >= out.capacity) continue;
        const DbObj& o = obj[i];
        out.label[rk] = o.label; out.npix[rk] = o.npix; out.flux_iso[rk] = o.flux;
        out.x[rk] = o.x; out.y[rk] = o.y; out.x2[rk] = o.x2; out.y2[rk] = o.y2; out.xy[rk] = o.xy;
        out.xmin[rk] = o.xmin; out.xmax[rk] = o.xmax; out.ymin[rk] = o.ymin; out.ymax[rk] = o.ymax;
        out.peak[rk] = o.peak; out.xpeak[rk] = o.xpeak; out.ypeak[rk] = o.ypeak; out.flags[rk] = o.flags;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *out.n = n;
}

cudaError_t launch_deblend(const Image& im, const SplineTab& sb, const SplineTab& sr, const float* taps, int kw,
                           int kh, float thresh, int minarea, int nthresh, float mincont, uint32_t* seg,
                           const gp_catalog& cat, const DeblendWork& w, const gp_catalog& objects, int* counts,
                           int* status, cudaStream_t st)
{
    DeblendArgs A;
    memset(&A, 0, sizeof A);
    A.im = im; A.sb = sb; A.sr = sr;
    A.kw = kw; A.kh = kh;
    for (int i = 0; i < kw * kh; ++i) A.taps[i] = taps[i];
    A.thresh = thresh; A.minarea = minarea; A.nthresh = nthresh; A.mincont = mincont;
    A.seg = seg;
    A.n_dev = cat.n; A.cap = cat.capacity;
    A.label = cat.label; A.npix = cat.npix;
    A.xmin = cat.xmin; A.xmax = cat.xmax; A.ymin = cat.ymin; A.ymax = cat.ymax;
    A.cand = w.cand; A.ctl = w.ctl; A.off = w.off;
    A.scratch = w.scratch;
    A.obj = w.obj; A.obj_count = w.ctl + DBC_OBJ; A.obj_stage_cap = w.obj_cap;
    A.counts = counts; A.status = status;
    cudaError_t e = cudaMemsetAsync(w.ctl, 0, DB_CTL * sizeof(int), st);
    if (e != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(counts, 0, 2 * sizeof(int), st)) != cudaSuccess) return e;
    const int grid = std::max(1, std::min((cat.capacity + 255) / 256, 152 * 8));
    k_db_select<<<grid, 256, 0, st>>>(cat.n, cat.capacity, cat.npix, cat.xmin, cat.xmax, cat.ymin, cat.ymax, minarea,
                                      kw / 2, kh / 2, w.cand, w.ctl, w.off);
    k_db_offsets<<<1, 1024, 0, st>>>(w.ctl, cat.capacity, w.off, w.scratch_bytes, status);
    auto* fn = im.is_f32 ? k_deblend<true> : k_deblend<false>;
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DB_SMEM)) != cudaSuccess) return e;
    fn<<<152, DB_NT, DB_SMEM, st>>>(A);
    k_db_place<<<grid, 256, 0, st>>>(w.obj, w.ctl + DBC_OBJ, w.obj_cap, objects);
    return cudaGetLastError();
}

}  // namespace gp
