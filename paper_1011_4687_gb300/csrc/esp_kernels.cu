// Staging, reduction and dispatch of the potential kernels for sm_103a.
//
// The potential kernels themselves are templates in esp_potential.cuh; each
// launch shape is compiled into its own object from esp_shape.cu, and the
// dispatchers below pick the shape's launcher.
#include "esp_potential.cuh"
#include "esp_shapes.h"

#include <cooperative_groups.h>

#include <algorithm>

namespace esp {

namespace {

// ---------------------------------------------------------------------------
// staging: recentre in FP64, split into FP32 hi + lo
// ---------------------------------------------------------------------------
// One recentred coordinate: its FP64 value, hi word on the environment's grid
// q (see the pair builder), lo word, and the rest in two words (esp_dd.h).
__device__ __forceinline__ void stage_coord(double x, double q, double iq, double *x64, float *xh, float *xl, float *xm,
                                            float *xr)
{
    float h, m, r;
    const double rest = dd_split3(x, q, iq, h, m, r);
    *x64 = x;
    *xh = h;
    *xl = (float)rest;
    *xm = m;
    *xr = r;
}

__device__ __forceinline__ void stage_position(const Staged &st, int j, double x, double y, double z, double q)
{
    const double iq = 1.0 / q;
    stage_coord(x, q, iq, st.x64 + j, st.xh + j, st.xl + j, st.xm + j, st.xr + j);
    stage_coord(y, q, iq, st.y64 + j, st.yh + j, st.yl + j, st.ym + j, st.yr + j);
    stage_coord(z, q, iq, st.z64 + j, st.zh + j, st.zl + j, st.zm + j, st.zr + j);
}

// slot_of (optional): the staged slot of position i (spatial order, below)
__global__ void stage_kernel(const double *__restrict__ pos, int n, double cx, double cy, double cz, double q,
                             Staged st, const int *__restrict__ slot_of)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const double *p = pos + 3 * (size_t)i; // (3 i passes 32 bits within the 2^30 positions of a call)
    double x = p[0] - cx, y = p[1] - cy, z = p[2] - cz;
    const int j = slot_of ? slot_of[i] : i;
    stage_position(st, j, x, y, z, q);
}

// ---------------------------------------------------------------------------
// spatial order of the positions: a stable counting sort by the Morton code
// of their cell in a 16^3 grid over [-8, 8]^3 bohr about the QM centre
// (positions outside share the edge cells).  A warp's positions then sit
// close together, so the warp-uniform far/near votes of the FP32C kernel
// follow the tiles' distance to that small region rather than to the whole
// QM sphere.  Deterministic: ties keep the input order.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int sort_cell(const double *__restrict__ pos, int i, double cx, double cy, double cz)
{
    const double *p = pos + 3 * (size_t)i;
    const double r[3] = {p[0] - cx, p[1] - cy, p[2] - cz};
    int key = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        int c = (int)floor((r[d] + kSortHalf) * (double(kSortSide) / (2.0 * kSortHalf)));
        c = min(max(c, 0), kSortSide - 1);
#pragma unroll
        for (int b = 0; b < 4; ++b)
            key |= ((c >> b) & 1) << (3 * b + d);
    }
    return key;
}

// The cell of every position.  Its own kernel over the whole GPU: at FP64's
// rate the cells of 65,536 positions take 2 us on 152 SMs and 30 us on the
// eight of the sort below.
__global__ void sort_key_kernel(const double *__restrict__ pos, int n, double cx, double cy, double cz,
                                int *__restrict__ key)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        key[i] = sort_cell(pos, i, cx, cy, cz);
}

__device__ __forceinline__ int warp_scan(int v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, v, o);
        v += lane >= o ? x : 0;
    }
    return v;
}

// Exclusive scan over the CTA of one value per thread (kSortThreads threads);
// part holds one int per warp.
__device__ __forceinline__ int cta_scan(int v, int *part)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int inc = warp_scan(v, lane);
    if (lane == 31)
        part[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const int p = part[lane];
        part[lane] = warp_scan(p, lane) - p;
    }
    __syncthreads();
    return part[warp] + inc - v;
}

// Stable scatter of positions [beg, end) by their cells key_slot[i], which the
// slots replace; run[c] is the next slot of cell c for this CTA.
__device__ __forceinline__ void cta_scatter(int *__restrict__ key_slot, int *__restrict__ perm, int beg, int end,
                                            int *run)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int base = beg; base < end; base += kSortThreads) {
        const int i = base + threadIdx.x;
        const bool valid = i < end;
        const int key = valid ? key_slot[i] : -1 - lane; // unique dummy keys
        const unsigned mask = __match_any_sync(0xffffffffu, key);
        const int rank = __popc(mask & lt);
        for (int w = 0; w < kSortThreads / 32; ++w) { // warps in order: ties keep the input order
            if (warp == w) {
                const bool leader = valid && rank == 0;
                int b0 = leader ? run[key] : 0;
                b0 = __shfl_sync(0xffffffffu, b0, __ffs(mask) - 1);
                if (leader)
                    run[key] = b0 + __popc(mask);
                if (valid) {
                    key_slot[i] = b0 + rank;
                    perm[b0 + rank] = i;
                }
            }
            __syncthreads();
        }
    }
}

// The order of all positions in one launch: a cluster of kSortCtas CTAs, each
// with the histogram of its contiguous part of the positions in shared memory;
// every CTA reads the others' histograms (distributed shared memory) for its
// own first slot in each cell.  (A histogram pass over up to 256 blocks, a scan
// of cells x blocks by one CTA and a scatter took 50 us for 10,000 positions
// and 257 us for 65,536, most of it the scan; now 14 us, and 30 for 50,000.)
__global__ void __cluster_dims__(kSortCtas, 1, 1) __launch_bounds__(kSortThreads)
    sort_cluster_kernel(int *__restrict__ key_slot, int n, int *__restrict__ perm)
{
    __shared__ __align__(16) int hist[kSortCells];
    __shared__ __align__(16) int run[kSortCells];
    __shared__ int part[32];
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = int(cl.block_rank()), t = threadIdx.x;
    const int chunk = (n + kSortCtas - 1) / kSortCtas;
    const int beg = min(n, rank * chunk), end = min(n, beg + chunk);
    constexpr int per = kSortCells / kSortThreads;
    static_assert(per == 4, "one int4 of cells per thread");
    reinterpret_cast<int4 *>(hist)[t] = make_int4(0, 0, 0, 0);
    __syncthreads();
    for (int i = beg + t; i < end; i += kSortThreads)
        atomicAdd(&hist[key_slot[i]], 1);
    cl.sync();
    int4 before = make_int4(0, 0, 0, 0), all = make_int4(0, 0, 0, 0);
#pragma unroll
    for (int r = 0; r < kSortCtas; ++r) {
        const int4 h = reinterpret_cast<const int4 *>(cl.map_shared_rank(hist, r))[t];
        all.x += h.x, all.y += h.y, all.z += h.z, all.w += h.w;
        if (r < rank)
            before.x += h.x, before.y += h.y, before.z += h.z, before.w += h.w;
    }
    const int first = cta_scan(all.x + all.y + all.z + all.w, part);
    int4 o;
    o.x = first + before.x;
    o.y = first + all.x + before.y;
    o.z = first + all.x + all.y + before.z;
    o.w = first + all.x + all.y + all.z + before.w;
    reinterpret_cast<int4 *>(run)[t] = o;
    cl.sync(); // (also: no CTA leaves while another still reads its histogram)
    cta_scatter(key_slot, perm, beg, end, run);
}

__global__ void batch_key_kernel(const BatchHeader *__restrict__ hdr, const SysDesc *__restrict__ sys)
{
    const int total = hdr->n_pos_total, n_sys = hdr->n_sys;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
        const SysDesc &d = sys[find_sys(sys, n_sys, g)];
        const int i = g - d.pos_begin;
        if (d.sorted)
            d.slot_of[i] = sort_cell(d.pos_in, i, d.qm[0], d.qm[1], d.qm[2]);
    }
}

__global__ void batch_stage_kernel(const BatchHeader *__restrict__ hdr, const SysDesc *__restrict__ sys)
{
    const int total = hdr->n_pos_total, n_sys = hdr->n_sys;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
        const SysDesc &d = sys[find_sys(sys, n_sys, g)];
        const int i = g - d.pos_begin;
        const double *p = d.pos_in + 3 * (size_t)i;
        double x = p[0] - d.qm[0], y = p[1] - d.qm[1], z = p[2] - d.qm[2];
        const int j = d.sorted ? d.slot_of[i] : i;
        stage_position(d.st, j, x, y, z, d.quantum);
    }
}

__global__ void batch_reduce_kernel(const BatchHeader *__restrict__ hdr, const SysDesc *__restrict__ sys)
{
    const int total = hdr->n_pos_total, n_sys = hdr->n_sys;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
        const SysDesc &d = sys[find_sys(sys, n_sys, g)];
        const int i = g - d.pos_begin;
        double s = 0.0, c = 0.0;
        if (d.n_tiles > 0)
            for (int k = 0; k < d.splits; ++k)
                two_sum_acc(s, c, d.partial[(size_t)k * d.n_pos + i]);
        d.V_out[d.sorted ? d.perm[i] : i] = s + c;
    }
}

// The spatial order of every sorted system of a batch, one CTA per system:
// histogram, scan and stable scatter as above, in its own shared memory.
__global__ void __launch_bounds__(kSortThreads) batch_sort_kernel(const BatchHeader *__restrict__ hdr,
                                                                  const SysDesc *__restrict__ sys)
{
    __shared__ __align__(16) int h[kSortCells];
    __shared__ int part[32];
    if ((int)blockIdx.x >= hdr->n_sys)
        return;
    const SysDesc &d = sys[blockIdx.x];
    if (!d.sorted)
        return;
    const int n = d.n_pos, t = threadIdx.x;
    reinterpret_cast<int4 *>(h)[t] = make_int4(0, 0, 0, 0);
    __syncthreads();
    for (int i = t; i < n; i += kSortThreads)
        atomicAdd(&h[d.slot_of[i]], 1);
    __syncthreads();
    const int4 v = reinterpret_cast<const int4 *>(h)[t];
    const int first = cta_scan(v.x + v.y + v.z + v.w, part);
    reinterpret_cast<int4 *>(h)[t] = make_int4(first, first + v.x, first + v.x + v.y, first + v.x + v.y + v.z);
    __syncthreads();
    cta_scatter(d.slot_of, d.perm, 0, n, h);
}

// ---------------------------------------------------------------------------
// few positions per call (the paper's call pattern: one r_new per Metropolis
// move).  The roles of the main kernels turn back to the paper's: threads
// take environment entries (cells, point charges, distributions) and evaluate
// them at the positions of their CTA's chunk (up to kSmallChunk of the n <=
// kSmallN positions; grid.y = chunk).  FP32 point charges are read in one flat
// coalesced pass over their contiguous records (each once per chunk), two
// positions per packed FP32 operation; the entries of the other tiles go to
// warps one tile half and one position at a time.  Every CTA writes its sums,
// and the last CTA of a chunk to finish adds them up in a fixed order.
//
// One launch, bound by its latency at one position (records from L2, two
// reductions) and by FP32 at many.  Before, 128-thread CTAs evaluated one
// position per operation, reduced every position over all lanes, put the
// nuclei's FP64 terms of all positions on one CTA and left the sum of 1,216
// partials to a second kernel: 268,818 cells at 1 / 16 / 128 positions took
// 18.4 / 39 / 78 us, now 9.8 / 16.6 / 37 (kernel).
// ---------------------------------------------------------------------------
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kNearList = 64;  // near entries a warp keeps for the end
constexpr int kNearDense = 24; // more of them in one item are evaluated at once

// (s, c) += (s2, c2) with the rounding error of s + s2 kept in c (TwoSum)
__device__ __forceinline__ void two_sum_pair(float &s, float &c, float s2, float c2)
{
    const float t = s + s2;
    const float bp = t - s;
    const float e = (s - (t - bp)) + (s2 - bp);
    s = t;
    c = (c + c2) + e;
}
__device__ __forceinline__ void two_sum_pair_xor(float &s, float &c, int o)
{
    const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
    two_sum_pair(s, c, s2, c2);
}

// Sums of NQ values per lane over the 32 lanes, halving the values with the
// lanes: lane l ends with the sum of value small_owner<NQ>(l).
template <int NQ>
__device__ __forceinline__ void warp_sums(float (&s)[NQ], float (&c)[NQ], int lane)
{
    int o = 16;
#pragma unroll
    for (int half = NQ / 2; half > 0; half >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const float so = up ? s[k] : s[k + half], co = up ? c[k] : c[k + half];
            const float s2 = __shfl_xor_sync(0xffffffffu, so, o), c2 = __shfl_xor_sync(0xffffffffu, co, o);
            s[k] = up ? s[k + half] : s[k];
            c[k] = up ? c[k + half] : c[k];
            two_sum_pair(s[k], c[k], s2, c2);
        }
    }
    for (; o > 0; o >>= 1)
        two_sum_pair_xor(s[0], c[0], o);
}
template <int NQ>
__device__ __forceinline__ int small_owner(int lane)
{
    int q = 0, o = 16;
#pragma unroll
    for (int half = NQ / 2; half > 0; half >>= 1, o >>= 1)
        q += lane & o ? half : 0;
    return q;
}

// one entry of a tile at one position, FP64
// (a call: its registers would spill those of the FP32 pass)
template <bool DIST>
__device__ __noinline__ double entry_f64(const SmallArgs &a, const TileMeta &m, int j, const double *p)
{
    if (!DIST || is_point_class(m.cls)) {
        const double *r = a.rec64 + m.off64 + (size_t)j * kPointStride64;
        const double dx = r[0] - p[0], dy = r[1] - p[1], dz = r[2] - p[2];
        return r[3] * esp_rsqrt(dx * dx + dy * dy + dz * dz);
    }
    return tile_f64_one_any(m.cls, a.rec64 + m.off64 + (size_t)j * rec64_stride(m.cls & 7), 1, p[0], p[1], p[2],
                            a.boys64);
}
// entries j, j + 1 where they exist
template <bool DIST>
__device__ __forceinline__ double entries_f64(const SmallArgs &a, const TileMeta &m, int j, const double *p)
{
    double v = 0.0;
    if (j < m.n)
        v = entry_f64<DIST>(a, m, j, p);
    if (j + 1 < m.n)
        v += entry_f64<DIST>(a, m, j + 1, p);
    return v;
}

// The same at FP64 accuracy with the far entries in FP32 words (as in
// potential_td_kernel, but two entries per lane); j differs by lane, the tile
// does not.
template <int L>
__device__ __noinline__ double far_pair(const DdTile t, int j, const DdPos &c, bool u0, bool u1, float *r2min)
{
    TdSum sum;
    sum.clear();
    f2 r2;
    td_far<L>(t, j, c, u0, u1, sum, r2);
    *r2min = fminf(r2.x, r2.y);
    return sum.total();
}
__device__ __noinline__ double point_pair(const DdTile t, int j, const DdPos &c, float *r2min)
{
    TdSum sum;
    sum.clear();
    f2 r2;
    td_point(t, j, c, sum, r2);
    *r2min = fminf(r2.x, r2.y);
    return sum.total();
}
// n0, n1: entries left to FP64.
template <bool DIST>
__device__ __forceinline__ double entries_words(const SmallArgs &a, const TileMeta &m, int j, const DdPos &c,
                                                bool &n0, bool &n1)
{
    const int n4 = dd_pad(m.n);
    const DdTile t = {a.recdd + (size_t)m.offdd * 4, n4};
    const bool mine = j < m.n;
    const float min_r2 = td_min_r2(a.dd_lim);
    double v = 0.0;
    float r2min = 1.0f;
    n0 = n1 = false;
    if (!DIST || is_point_class(m.cls)) {
        if (mine)
            v = point_pair(t, j, c, &r2min);
    } else if constexpr (DIST) {
        if (mine) {
            const f2 dx = t(0, j) - f2(c.h[0]), dy = t(1, j) - f2(c.h[1]), dz = t(2, j) - f2(c.h[2]);
            const f2 s = esp_fma(dx, dx, esp_fma(dy, dy, dz * dz)), T = t(10, j) * s;
            n0 = !td_is_far(T.x, s.x, min_r2);
            n1 = !td_is_far(T.y, s.y, min_r2);
            switch (m.cls & 7) {
            case 0: v = far_pair<0>(t, j, c, !n0, !n1, &r2min); break;
            case 1: v = far_pair<1>(t, j, c, !n0, !n1, &r2min); break;
            case 2: v = far_pair<2>(t, j, c, !n0, !n1, &r2min); break;
            case 3: v = far_pair<3>(t, j, c, !n0, !n1, &r2min); break;
            default: v = far_pair<4>(t, j, c, !n0, !n1, &r2min); break;
            }
        }
    }
    if (!(r2min >= min_r2)) { // closer than the words resolve
        v = 0.0;
        n0 = n1 = true;
    }
    n0 &= mine;
    n1 &= j + 1 < m.n;
    return v;
}

// the words of two positions
struct PairPos {
    f2 xh, yh, zh, xl, yl, zl;
    __device__ __forceinline__ explicit PairPos(const float *s)
    {
        const float4 a = reinterpret_cast<const float4 *>(s)[0], b = reinterpret_cast<const float4 *>(s)[1],
                     c = reinterpret_cast<const float4 *>(s)[2];
        xh = f2(a.x, a.y), yh = f2(a.z, a.w), zh = f2(b.x, b.y);
        xl = f2(b.z, b.w), yl = f2(c.x, c.y), zl = f2(c.z, c.w);
    }
};
// one FP32 point charge
struct P32Entry {
    f2 xh, yh, zh, xl, yl, zl, qh, ql;
    __device__ __forceinline__ explicit P32Entry(const float *__restrict__ r)
    {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(r));
        const float4 b = __ldg(reinterpret_cast<const float4 *>(r) + 1);
        xh = f2(a.x), yh = f2(a.y), zh = f2(a.z), xl = f2(b.x), yl = f2(b.y), zl = f2(b.z);
        qh = f2(__ldg(r + rec32_m(0))), ql = f2(b.w);
    }
    __device__ __forceinline__ f2 term(const PairPos &p) const
    {
        const f2 dx = (xh - p.xh) + (xl - p.xl), dy = (yh - p.yh) + (yl - p.yl), dz = (zh - p.zh) + (zl - p.zl);
        const f2 rs = esp_rsqrt(esp_fma(dx, dx, esp_fma(dy, dy, dz * dz)));
        return esp_fma(qh, rs, ql * rs);
    }
};

// What a kernel holds besides the FP32 point charges: point charges alone;
// distributions, all of them in FP64 (direct); distributions in words.  Up to four
// positions take 64 registers and two CTAs per SM; the words' code, whose calls made
// every thread spill there (a stack of 424 bytes), takes 128 and one (1 x 96,000
// products and their FP32 points: 31 us with the words' code aboard, 27 direct).
enum SmallMode { kSmallPoints, kSmallDirect, kSmallWords };
constexpr int small_ctas(int nq, int mode) { return nq <= 4 && mode != kSmallWords ? 2 : 1; }
template <int NQ, int MODE>
__global__ void __launch_bounds__(kSmallThreads, small_ctas(NQ, MODE))
    small_n_kernel(SmallArgs a, double *__restrict__ V)
{
    // grid: x = slice of the environment's entries, y = chunk of positions
    constexpr bool DIST = MODE != kSmallPoints;
    __shared__ double s_pos[NQ][3];
    __shared__ DdPos s_dd[NQ];
    __shared__ __align__(16) float s_pair[NQ / 2 > 0 ? NQ / 2 : 1][12]; // lanes' hi x y z, lo x y z of position pairs
    __shared__ float2 s_red[kSmallWarps][NQ]; // sums in FP32 with compensation
    __shared__ double s_red64[kSmallWarps][NQ];
    __shared__ int2 s_list[kSmallWarps][kNearList]; // tile, entry * kSmallChunk + position
    __shared__ double s_val[kSmallWarps * kNearList];
    __shared__ unsigned char s_own[kSmallWarps * kNearList];
    __shared__ int s_listed[kSmallWarps];
    __shared__ int s_last;
    const int n = a.n_pos, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int q0 = blockIdx.y * kSmallChunk;
    const int nq = min(NQ, n - q0);
    // does this CTA take any entry in FP64 (or as dd sums)?
    const int units = a.n_other * a.tile_parts;
    const bool has64 = int(blockIdx.x) < units;
    if (t < 3 * NQ) {
        const int q = min(t / 3, nq - 1), d = t % 3; // (padding repeats the last position)
        const double x = a.pos_in[3 * (q0 + q) + d] - (d == 0 ? a.cx : d == 1 ? a.cy : a.cz);
        float h, m, r;
        const double rest = dd_split3(x, a.quantum, a.inv_quantum, h, m, r);
        s_pos[t / 3][d] = x;
        s_dd[t / 3].h[d] = h;
        s_dd[t / 3].m[d] = m;
        s_dd[t / 3].l[d] = r;
        s_pair[t / 6][2 * d + (t / 3) % 2] = h;
        s_pair[t / 6][6 + 2 * d + (t / 3) % 2] = float(rest);
    }
    if (t < kSmallWarps * NQ) {
        s_red[t / NQ][t % NQ] = make_float2(0.0f, 0.0f);
        s_red64[t / NQ][t % NQ] = 0.0;
    }
    __syncthreads();
    // FP32 point charges: thread g takes entries g, g + G, ... (the paper's
    // coalesced mapping) and sums its terms in FP32
    const int g0 = blockIdx.x * kSmallThreads + t;
    if (a.n_p32 > 0) {
        constexpr int NP = NQ / 2;
        f2 acc[NP];
#pragma unroll
        for (int k = 0; k < NP; ++k)
            acc[k] = f2(0.0f);
        if (g0 < a.g_threads) {
            const float *rec = a.rec32 + a.p32_off;
            const size_t step = (size_t)a.g_threads * rec32_stride(0);
            const float *r = rec + (size_t)g0 * rec32_stride(0);
            int e = g0;
            // two entries per pass over the positions (their words come from
            // shared memory once for both), each sum in the entries' order
            for (; e + a.g_threads < a.n_p32; e += 2 * a.g_threads, r += 2 * step) {
                const P32Entry u(r), v(r + step);
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    const PairPos p(s_pair[k]);
                    const f2 x = u.term(p), y = v.term(p);
                    acc[k] += x;
                    acc[k] += y;
                }
            }
            if (e < a.n_p32) {
                const P32Entry u(r);
#pragma unroll
                for (int k = 0; k < NP; ++k)
                    acc[k] += u.term(PairPos(s_pair[k]));
            }
        }
        float s[NQ], c[NQ];
#pragma unroll
        for (int k = 0; k < NQ; ++k) {
            s[k] = k % 2 ? acc[k / 2].y : acc[k / 2].x;
            c[k] = 0.0f;
        }
        warp_sums<NQ>(s, c, lane);
        s_red[warp][small_owner<NQ>(lane)] = make_float2(s[0], c[0]); // (lanes of one owner hold the same sum)
        __syncwarp();
    }
    // the other tiles: CTA b takes the parts b, b + grid, ..., its warps one
    // (part, position) item after the other, two entries per lane
    if (has64) {
        int listed = 0; // entries in this warp's list
        const int my_units = (units - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x);
        for (int item = warp; item < my_units * nq; item += kSmallWarps) {
            const int u = blockIdx.x + gridDim.x * (item / nq), q = item % nq;
            const int o = u / a.tile_parts;
            const int tile = o < a.skip_begin ? o : o + a.n_skip;
            const TileMeta m = a.tiles[tile];
            const int j = a.direct ? (u % a.tile_parts) * 32 + lane : (u % a.tile_parts) * 64 + 2 * lane;
            const bool words = m.offdd >= 0 && dd_in_range(s_dd[q].h, a.dd_lim);
            if (MODE == kSmallDirect || (MODE == kSmallPoints && a.direct)) { // (FP64 throughout)
                double v = j < m.n ? entry_f64<DIST>(a, m, j, s_pos[q]) : 0.0;
#pragma unroll
                for (int w = 16; w > 0; w >>= 1)
                    v += __shfl_xor_sync(0xffffffffu, v, w);
                if (lane == 0)
                    s_red64[warp][q] += v;
            } else if (m.cls == kClassPoint && a.points_dd) {
                // beside FP32 sums: dd sums
                float s = 0.0f, c = 0.0f;
                if (j < m.n) {
                    const DdTile tile = {a.recdd + (size_t)m.offdd * 4, dd_pad(m.n)};
                    f2 r2;
                    const dd v = dd_point(tile, j, s_dd[q], r2);
                    s = v.h.x, c = v.l.x;
                    two_sum_pair(s, c, v.h.y, v.l.y); // (a padding charge is zero)
                    if (!(fminf(r2.x, r2.y) >= dd_min_r2(a.dd_lim)) || !words) {
                        const double x = entries_f64<DIST>(a, m, j, s_pos[q]);
                        s = float(x);
                        c = float(x - double(s));
                    }
                }
#pragma unroll
                for (int w = 16; w > 0; w >>= 1)
                    two_sum_pair_xor(s, c, w);
                if (lane == 0) {
                    float2 x = s_red[warp][q];
                    two_sum_pair(x.x, x.y, s, c);
                    s_red[warp][q] = x;
                }
            } else {
                double v = 0.0;
                bool n0 = j < m.n, n1 = j + 1 < m.n;
                if constexpr (MODE != kSmallDirect)
                    if (words && td_resolves(a.dd_lim))
                        v = entries_words<DIST>(a, m, j, s_dd[q], n0, n1);
                // near entries: an FP64 operation takes its 64 cycles whatever
                // the number of lanes, so few of them wait in the warp's list
                const unsigned b0 = __ballot_sync(0xffffffffu, n0), b1 = __ballot_sync(0xffffffffu, n1);
                const int c0 = __popc(b0), cnt = c0 + __popc(b1);
                if (cnt <= kNearDense && listed + cnt <= kNearList) {
                    const unsigned below = (1u << lane) - 1u;
                    if (n0)
                        s_list[warp][listed + __popc(b0 & below)] = make_int2(tile, j * kSmallChunk + q);
                    if (n1)
                        s_list[warp][listed + c0 + __popc(b1 & below)] = make_int2(tile, (j + 1) * kSmallChunk + q);
                    listed += cnt;
                } else {
                    if (n0)
                        v += entry_f64<DIST>(a, m, j, s_pos[q]);
                    if (n1)
                        v += entry_f64<DIST>(a, m, j + 1, s_pos[q]);
                }
#pragma unroll
                for (int w = 16; w > 0; w >>= 1)
                    v += __shfl_xor_sync(0xffffffffu, v, w);
                if (lane == 0)
                    s_red64[warp][q] += v;
            }
            __syncwarp();
        }
        if (lane == 0)
            s_listed[warp] = listed;
        __syncthreads();
        // the listed entries, one per thread, then each position's values by its warp
        int total = 0;
        for (int w = 0; w < kSmallWarps; ++w)
            total += s_listed[w];
        for (int k = t; k < total; k += kSmallThreads) {
            int w = 0, i = k;
            while (i >= s_listed[w])
                i -= s_listed[w++];
            const int2 x = s_list[w][i];
            const TileMeta m = a.tiles[x.x];
            s_val[k] = entry_f64<DIST>(a, m, x.y / kSmallChunk, s_pos[x.y % kSmallChunk]);
            s_own[k] = (unsigned char)(x.y % kSmallChunk);
        }
        __syncthreads();
        if (warp < nq && total > 0) {
            double v = 0.0;
            for (int k = lane; k < total; k += 32)
                if (s_own[k] == warp)
                    v += s_val[k];
#pragma unroll
            for (int w = 16; w > 0; w >>= 1)
                v += __shfl_xor_sync(0xffffffffu, v, w);
            if (lane == 0)
                s_red64[warp][warp] += v; // (row warp: only this thread adds to it now)
        }
    }
    __syncthreads();
    // this CTA's sums, warps in order
    float2 *part32 = a.part32 + (size_t)blockIdx.y * gridDim.x * NQ;
    double *part64 = a.part64 + (size_t)blockIdx.y * gridDim.x * NQ;
    if (t < NQ) {
        float2 x = s_red[0][t];
        double v = s_red64[0][t];
        for (int w = 1; w < kSmallWarps; ++w) {
            two_sum_pair(x.x, x.y, s_red[w][t].x, s_red[w][t].y);
            if (has64 && a.any64)
                v += s_red64[w][t];
        }
        part32[blockIdx.x * NQ + t] = x;
        if (has64 && a.any64)
            part64[blockIdx.x * NQ + t] = v;
        __threadfence();
    }
    __syncthreads();
    if (t == 0)
        s_last = atomicAdd(&a.counters[blockIdx.y], 1) == int(gridDim.x) - 1;
    __syncthreads();
    if (!s_last)
        return;
    // last CTA of the chunk: thread t takes position t % NQ of the slices t / NQ, ...
    __threadfence();
    const int n64 = a.any64 ? min(units, int(gridDim.x)) : 0;
    constexpr int rows = kSmallThreads / NQ;
    const int q = t % NQ;
    float s = 0.0f, c = 0.0f;
    for (int k = t / NQ; k < int(gridDim.x); k += rows) {
        const float2 x = __ldcg(part32 + (size_t)k * NQ + q);
        two_sum_pair(s, c, x.x, x.y);
    }
    double s64 = 0.0, c64 = 0.0;
    for (int k = t / NQ; k < n64; k += rows)
        two_sum_acc(s64, c64, __ldcg(part64 + (size_t)k * NQ + q));
    // the warp's lanes of one position, then the warps
#pragma unroll
    for (int o = 16; o >= NQ; o >>= 1) {
        two_sum_pair_xor(s, c, o);
        if (n64 > 0) {
            const double a2 = __shfl_xor_sync(0xffffffffu, s64, o), b2 = __shfl_xor_sync(0xffffffffu, c64, o);
            two_sum_acc(s64, c64, a2);
            c64 += b2;
        }
    }
    __shared__ double s_fin[kSmallWarps][NQ][2];
    __syncthreads();
    if (lane < NQ) {
        s_red[warp][lane] = make_float2(s, c);
        s_fin[warp][lane][0] = s64;
        s_fin[warp][lane][1] = c64;
    }
    __syncthreads();
    if (warp < nq) { // warp q: position q, lane w the sums of warp w
        float2 x = lane < kSmallWarps ? s_red[lane][warp] : make_float2(0.0f, 0.0f);
        double v = 0.0, w = 0.0;
        if (n64 > 0 && lane < kSmallWarps) {
            v = s_fin[lane][warp][0];
            w = s_fin[lane][warp][1];
        }
#pragma unroll
        for (int o = kSmallWarps / 2; o > 0; o >>= 1) {
            two_sum_pair_xor(x.x, x.y, o);
            if (n64 > 0) {
                const double v2 = __shfl_xor_sync(0xffffffffu, v, o), w2 = __shfl_xor_sync(0xffffffffu, w, o);
                two_sum_acc(v, w, v2);
                w += w2;
            }
        }
        if (lane == 0) {
            const double y = double(x.x) + double(x.y);
            V[q0 + warp] = n64 > 0 ? y + (v + w) : y;
        }
    }
    if (t == 0)
        a.counters[blockIdx.y] = 0; // for the next call
}

// ---------------------------------------------------------------------------
// reductions
// ---------------------------------------------------------------------------
// (s, c) += (s2, c2)
__device__ __forceinline__ void two_sum_join(double &s, double &c, double s2, double c2)
{
    two_sum_acc(s, c, s2);
    c += c2;
}

// V of 32 positions per CTA: warp y sums the partials y, y + SLICES, ... of its
// lanes' positions by TwoSum, then the slices are joined in a fixed order.
// Bound by the latency of the FP64 additions: one thread per position took 25
// us for 39 partials of 10,000 positions and 64 us for 57 of 65,536.
// perm (optional): the input index of staged slot i
template <int SLICES>
__global__ void __launch_bounds__(32 * SLICES) reduce_kernel(const double *__restrict__ partial, int n_splits, int n,
                                                              double *__restrict__ V, const int *__restrict__ perm)
{
    __shared__ double s_s[SLICES][32], s_c[SLICES][32];
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + x;
    double s = 0.0, c = 0.0;
    if (i < n) {
#pragma unroll 4
        for (int k = y; k < n_splits; k += SLICES)
            two_sum_acc(s, c, partial[(size_t)k * n + i]);
    }
    s_s[y][x] = s;
    s_c[y][x] = c;
#pragma unroll
    for (int o = SLICES / 2; o > 0; o >>= 1) {
        __syncthreads();
        if (y < o) {
            two_sum_join(s, c, s_s[y + o][x], s_c[y + o][x]);
            s_s[y][x] = s;
            s_c[y][x] = c;
        }
    }
    if (y == 0 && i < n)
        V[perm ? perm[i] : i] = s + c;
}

// The same where the partials after the first n64 (the dd kernel's, FP64) are
// FP32 (sum, compensation) pairs, as an FP32C kernel holds them: few FP64
// operations (FP64 partials of 1,001 positions in 512 splits took 38 us, of
// 65,536 in 60 splits 65 us; now 7 us, and 25 for 50,000 in 68).
template <int SLICES>
__global__ void __launch_bounds__(32 * SLICES) reduce_pairs_kernel(const double *__restrict__ partial, int n64,
                                                                    int n_splits, int n, double *__restrict__ V,
                                                                    const int *__restrict__ perm)
{
    __shared__ float2 s_p[SLICES][32];
    __shared__ double s_s[SLICES][32], s_c[SLICES][32];
    const float2 *pairs = reinterpret_cast<const float2 *>(partial);
    const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + x;
    float s = 0.0f, c = 0.0f;
    double s64 = 0.0, c64 = 0.0;
    if (i < n) {
        for (int k = y; k < n64; k += SLICES)
            two_sum_acc(s64, c64, partial[(size_t)k * n + i]);
#pragma unroll 4
        for (int k = n64 + y; k < n_splits; k += SLICES) {
            const float2 p = pairs[(size_t)k * n + i];
            two_sum_pair(s, c, p.x, p.y);
        }
    }
    s_p[y][x] = make_float2(s, c);
    s_s[y][x] = s64;
    s_c[y][x] = c64;
#pragma unroll
    for (int o = SLICES / 2; o > 0; o >>= 1) {
        __syncthreads();
        if (y < o) {
            two_sum_pair(s, c, s_p[y + o][x].x, s_p[y + o][x].y);
            s_p[y][x] = make_float2(s, c);
            if (y + o < n64) { // (slices from n64 on hold no FP64 partial)
                two_sum_join(s64, c64, s_s[y + o][x], s_c[y + o][x]);
                s_s[y][x] = s64;
                s_c[y][x] = c64;
            }
        }
    }
    if (y == 0 && i < n)
        V[perm ? perm[i] : i] = (s64 + c64) + (double(s) + double(c));
}

// one warp per walker: its lanes' electrons by TwoSum, then the lanes in a fixed order
__global__ void walker_kernel(const double *__restrict__ V, int n_walkers, int n_elec, double *__restrict__ E)
{
    // (blocks first: 32 n_walkers threads pass 2^32 from 2^27 walkers on)
    const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (w >= n_walkers)
        return;
    double s = 0.0, c = 0.0;
    for (int e = lane; e < n_elec; e += 32)
        two_sum_acc(s, c, -V[(size_t)w * n_elec + e]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double s2 = __shfl_down_sync(0xffffffffu, s, o), c2 = __shfl_down_sync(0xffffffffu, c, o);
        two_sum_join(s, c, s2, c2);
    }
    if (lane == 0)
        E[w] = s + c;
}

} // namespace

bool potential_shape_supported(int precision, int threads, int ppt)
{
#define ESP_SHAPE_IS(NT, PPT) || (threads == NT && ppt == PPT)
    if (precision == 0)
        return false ESP_F64_SHAPES(ESP_SHAPE_IS);
    return false ESP_F32C_SHAPES(ESP_SHAPE_IS);
#undef ESP_SHAPE_IS
}

size_t potential_smem_bytes(int precision, int tile_size)
{
    if (precision == 0)
        return (size_t)tile_size * 40 * sizeof(double);
    return (size_t)tile_size * kRec32MaxStride * sizeof(float) + (size_t)kBoys32Rows * kBoys32Row * sizeof(float);
}

cudaError_t launch_stage(const double *pos_in, int n, const double center[3], double quantum, const Staged &st,
                         cudaStream_t s, const int *slot_of)
{
    if (n <= 0)
        return cudaSuccess;
    stage_kernel<<<(n + 255) / 256, 256, 0, s>>>(pos_in, n, center[0], center[1], center[2], quantum, st, slot_of);
    return cudaGetLastError();
}

size_t sort_scratch_ints(int n) { return 2 * (size_t)n; }

cudaError_t launch_sort(const double *pos_in, int n, const double center[3], int *scratch, int **slot_of, int **perm,
                        cudaStream_t s)
{
    *slot_of = scratch;
    *perm = scratch + n;
    sort_key_kernel<<<(n + 127) / 128, 128, 0, s>>>(pos_in, n, center[0], center[1], center[2], *slot_of);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    sort_cluster_kernel<<<kSortCtas, kSortThreads, 0, s>>>(*slot_of, n, *perm);
    return cudaGetLastError();
}

cudaError_t launch_potential(int precision, const EvalArgs &a, int threads, int ppt, cudaStream_t s)
{
    if (a.n_pos <= 0)
        return cudaSuccess;
    const int per_cta = threads * ppt;
    dim3 grid((a.n_pos + per_cta - 1) / per_cta, a.n_splits);
    size_t smem = potential_smem_bytes(precision, a.tile_size);
#define ESP_LAUNCH_F64(NT, PPT) \
    if (threads == NT && ppt == PPT) return launch_f64_shape<NT, PPT>(a, grid, smem, s);
#define ESP_LAUNCH_F32C(NT, PPT) \
    if (threads == NT && ppt == PPT) return launch_f32c_shape<NT, PPT>(a, grid, smem, s);
    if (precision == 0) {
        ESP_F64_SHAPES(ESP_LAUNCH_F64)
    } else {
        ESP_F32C_SHAPES(ESP_LAUNCH_F32C)
    }
#undef ESP_LAUNCH_F64
#undef ESP_LAUNCH_F32C
    return cudaErrorInvalidConfiguration;
}

cudaError_t launch_batch(int precision, const BatchHeader *hdr, const SysDesc *sys, const BatchGroup *groups,
                         int max_sys, int *counter,
                         int max_items, const float *boys32, const double *boys64, const float *boysdd, int tile_cap,
                         int threads, int ppt,
                         int num_sms, int max_pos_total, cudaStream_t s)
{
    const int sgrid = std::max(1, std::min(4 * num_sms, (max_pos_total + 255) / 256));
    batch_key_kernel<<<sgrid, 256, 0, s>>>(hdr, sys);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    batch_sort_kernel<<<std::max(1, max_sys), kSortThreads, 0, s>>>(hdr, sys);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    batch_stage_kernel<<<sgrid, 256, 0, s>>>(hdr, sys);
    e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    const size_t smem = potential_smem_bytes(precision, tile_cap);
    bool launched = false;
#define ESP_BLAUNCH(NT, PPT, PR)                                                                                \
    if (!launched && threads == NT && ppt == PPT && precision == PR) {                                        \
        e = launch_batch_shape<NT, PPT, PR>(hdr, sys, groups, counter, max_items, boys32, boys64, boysdd, tile_cap, num_sms, smem, \
                                            s); \
        launched = true;                                                                                      \
    }
    ESP_BATCH_SHAPES(ESP_BLAUNCH)
#undef ESP_BLAUNCH
    if (!launched)
        return cudaErrorInvalidConfiguration;
    if (e != cudaSuccess)
        return e;
    batch_reduce_kernel<<<sgrid, 256, 0, s>>>(hdr, sys);
    return cudaGetLastError();
}

bool batch_shape_supported(int precision, int threads, int ppt)
{
#define ESP_BSHAPE_IS(NT, PPT, PR) || (threads == NT && ppt == PPT && precision == PR)
    return false ESP_BATCH_SHAPES(ESP_BSHAPE_IS);
#undef ESP_BSHAPE_IS
}

// The sums of one thread: entries g, g + G, ... of the FP32 point charges, G =
// 128 threads for each of about 8 slices per SM over all chunks of positions,
// so that with more positions each thread takes more entries and the
// per-position reductions are amortised over more terms.
int small_n_threads(int n_tiles, int num_sms, int n)
{
    const int chunks = std::max(1, (n + kSmallChunk - 1) / kSmallChunk);
    return 128 * std::max(1, std::min(n_tiles, 8 * num_sms / chunks));
}

namespace {

// positions a chunk holds: two (one pair) up to kSmallChunk
int small_nq(int n) { return n <= 2 ? 2 : n <= 4 ? 4 : n <= 8 ? 8 : 16; }

// CTAs of a chunk: its FP32 threads; without FP32 entries one CTA per SM over
// all chunks (5 positions x 889 tiles: 223 CTAs, a second wave of 71, took 50 us)
int small_grid(int g_threads, int num_sms, int chunks, bool fp32)
{
    const int grid = (g_threads + kSmallThreads - 1) / kSmallThreads;
    return fp32 ? grid : std::min(grid, std::max(1, num_sms / chunks));
}

} // namespace

size_t small_n_bytes(int n_tiles, int num_sms, int n)
{
    const int chunks = std::max(1, (n + kSmallChunk - 1) / kSmallChunk);
    const int grid = std::max(small_grid(small_n_threads(n_tiles, num_sms, n), num_sms, chunks, true), num_sms / chunks);
    return (size_t)grid * chunks * small_nq(n) * (sizeof(float2) + sizeof(double));
}

cudaError_t launch_small_n(SmallArgs a, void *scratch, int num_sms, double *V, cudaStream_t s)
{
    if (a.n_pos <= 0 || a.n_pos > kSmallN)
        return cudaErrorInvalidValue;
    a.g_threads = small_n_threads(a.n_tiles, num_sms, a.n_pos);
    const int nq = small_nq(a.n_pos);
    const int chunks = (a.n_pos + kSmallChunk - 1) / kSmallChunk;
    const int mode = !a.dist ? kSmallPoints : a.direct ? kSmallDirect : kSmallWords;
    // one CTA per SM, where each thread has one FP32 entry at most all the same
    const int per_wave = num_sms / chunks * kSmallThreads;
    if (mode == kSmallWords && a.n_p32 <= per_wave)
        a.g_threads = std::min(a.g_threads, per_wave);
    dim3 grid(small_grid(a.g_threads, num_sms, chunks, a.n_p32 > 0), chunks);
    if (a.direct) // latency counts: a part per CTA
        grid.x = std::max(int(grid.x), std::min(a.n_other * a.tile_parts, num_sms / chunks));
    a.part64 = static_cast<double *>(scratch);
    a.part32 = reinterpret_cast<float2 *>(a.part64 + (size_t)grid.x * grid.y * nq);
#define ESP_SMALL(NQ)                                                           \
    if (mode == kSmallWords)                                                    \
        small_n_kernel<NQ, kSmallWords><<<grid, kSmallThreads, 0, s>>>(a, V);   \
    else if (mode == kSmallDirect)                                              \
        small_n_kernel<NQ, kSmallDirect><<<grid, kSmallThreads, 0, s>>>(a, V);  \
    else                                                                        \
        small_n_kernel<NQ, kSmallPoints><<<grid, kSmallThreads, 0, s>>>(a, V)
    switch (nq) {
    case 2: ESP_SMALL(2); break;
    case 4: ESP_SMALL(4); break;
    case 8: ESP_SMALL(8); break;
    default: ESP_SMALL(16); break;
    }
#undef ESP_SMALL
    return cudaGetLastError();
}

cudaError_t launch_reduce(const double *partial, int n_splits, int n, double *V, cudaStream_t s, const int *perm,
                          bool in_order, int n64)
{
    if (n <= 0)
        return cudaSuccess;
    const int grid = (n + 31) / 32;
    // more slices where the partials are many and the positions few
    if (n64 >= 0 && n_splits > 64)
        reduce_pairs_kernel<32><<<grid, 32 * 32, 0, s>>>(partial, n64, n_splits, n, V, perm);
    else if (n64 >= 0)
        reduce_pairs_kernel<8><<<grid, 32 * 8, 0, s>>>(partial, n64, n_splits, n, V, perm);
    else if (in_order)
        reduce_kernel<1><<<grid, 32, 0, s>>>(partial, n_splits, n, V, perm);
    else if (n_splits > 64)
        reduce_kernel<32><<<grid, 32 * 32, 0, s>>>(partial, n_splits, n, V, perm);
    else
        reduce_kernel<8><<<grid, 32 * 8, 0, s>>>(partial, n_splits, n, V, perm);
    return cudaGetLastError();
}

cudaError_t launch_walkers(const double *V, int n_walkers, int n_elec, double *E, cudaStream_t s)
{
    if (n_walkers <= 0)
        return cudaSuccess;
    walker_kernel<<<(n_walkers + 3) / 4, 128, 0, s>>>(V, n_walkers, n_elec, E);
    return cudaGetLastError();
}

} // namespace esp
