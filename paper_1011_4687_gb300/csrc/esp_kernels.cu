// Staging, reduction and dispatch of the potential kernels for sm_103a.
//
// The potential kernels themselves are templates in esp_potential.cuh; each
// launch shape is compiled into its own object from esp_shape.cu, and the
// dispatchers below pick the shape's launcher.
#include "esp_dd.h"
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
__device__ __forceinline__ void stage_coord(double x, double q, double *x64, float *xh, float *xl, float *xm,
                                            float *xr)
{
    float h, m, r;
    const double rest = dd_split3(x, q, h, m, r);
    *x64 = x;
    *xh = h;
    *xl = (float)rest;
    *xm = m;
    *xr = r;
}

__device__ __forceinline__ void stage_position(const Staged &st, int j, double x, double y, double z, double q)
{
    stage_coord(x, q, st.x64 + j, st.xh + j, st.xl + j, st.xm + j, st.xr + j);
    stage_coord(y, q, st.y64 + j, st.yh + j, st.yl + j, st.ym + j, st.yr + j);
    stage_coord(z, q, st.z64 + j, st.zh + j, st.zl + j, st.zm + j, st.zr + j);
}

// slot_of (optional): the staged slot of position i (spatial order, below)
__global__ void stage_kernel(const double *__restrict__ pos, int n, double cx, double cy, double cz, double q,
                             Staged st, const int *__restrict__ slot_of)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    double x = pos[3 * i] - cx, y = pos[3 * i + 1] - cy, z = pos[3 * i + 2] - cz;
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
    const double r[3] = {pos[3 * i] - cx, pos[3 * i + 1] - cy, pos[3 * i + 2] - cz};
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
// and 257 us for 65,536, most of it the scan.)
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
        const SysDesc &d = sys[find_sys(sys, n_sys, g, false)];
        const int i = g - d.pos_begin;
        if (d.sorted)
            d.slot_of[i] = sort_cell(d.pos_in, i, d.qm[0], d.qm[1], d.qm[2]);
    }
}

__global__ void batch_stage_kernel(const BatchHeader *__restrict__ hdr, const SysDesc *__restrict__ sys)
{
    const int total = hdr->n_pos_total, n_sys = hdr->n_sys;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
        const SysDesc &d = sys[find_sys(sys, n_sys, g, false)];
        const int i = g - d.pos_begin;
        double x = d.pos_in[3 * i] - d.qm[0], y = d.pos_in[3 * i + 1] - d.qm[1], z = d.pos_in[3 * i + 2] - d.qm[2];
        const int j = d.sorted ? d.slot_of[i] : i;
        stage_position(d.st, j, x, y, z, d.quantum);
    }
}

__global__ void batch_reduce_kernel(const BatchHeader *__restrict__ hdr, const SysDesc *__restrict__ sys)
{
    const int total = hdr->n_pos_total, n_sys = hdr->n_sys;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
        const SysDesc &d = sys[find_sys(sys, n_sys, g, false)];
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
// kSmallN positions; grid.y = chunk), the CTA reduces per position in a fixed
// order, and CTA (b, chunk) writes partial[b][q] for its chunk's q.  FP32
// point charges are read in one flat coalesced pass over their contiguous
// records (each once per chunk); the other tiles are dealt round-robin to the
// CTAs of a chunk and read from the FP64 records.
// ---------------------------------------------------------------------------
constexpr int kSmallThreads = 128;

// (s, c) += (s2, c2) with the rounding error of s + s2 kept in c (TwoSum)
__device__ __forceinline__ void two_sum_pair(float &s, float &c, float s2, float c2)
{
    const float t = s + s2;
    const float bp = t - s;
    const float e = (s - (t - bp)) + (s2 - bp);
    s = t;
    c = (c + c2) + e;
}

__global__ void __launch_bounds__(kSmallThreads, 4) small_n_kernel(SmallArgs a)
{
    // grid: x = slice of the environment's entries, y = chunk of kSmallChunk
    // positions; each (slice, position) partial sum is written by one CTA
    __shared__ double s_pos[kSmallChunk][3];
    __shared__ float s_ph[kSmallChunk][3], s_pl[kSmallChunk][3]; // FP32 hi (on the records' grid) and lo words
    __shared__ float s_red32[kSmallThreads / 32][kSmallChunk][2];
    __shared__ double s_red64[kSmallThreads / 32][kSmallChunk];
    const int n = a.n_pos;
    const int q0 = blockIdx.y * kSmallChunk;
    const int nq = min(kSmallChunk, n - q0);
    for (int i = threadIdx.x; i < nq * 3; i += kSmallThreads) {
        const int c = i % 3;
        const double x = a.pos_in[3 * q0 + i] - (c == 0 ? a.cx : c == 1 ? a.cy : a.cz);
        const double h = nearbyint(x / a.quantum) * a.quantum;
        s_pos[i / 3][c] = x;
        s_ph[i / 3][c] = float(h);
        s_pl[i / 3][c] = float(x - h);
    }
    // does this CTA evaluate any entry in FP64?  (then its FP64 sums need a
    // FP64 reduction; FP64 instructions run at 1/64 of the FP32 rate here)
    bool has64 = false;
    for (int t = blockIdx.x; t < a.n_tiles && !has64; t += gridDim.x)
        has64 = !(a.tiles[t].cls == kClassPoint32 && a.fp32);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gtid = blockIdx.x * kSmallThreads + threadIdx.x, gthreads = gridDim.x * kSmallThreads;
    float acc32[kSmallChunk];
    double acc[kSmallChunk];
#pragma unroll
    for (int q = 0; q < kSmallChunk; ++q) {
        acc32[q] = 0.0f;
        acc[q] = 0.0;
    }
    // FP32 point charges: one flat, coalesced pass over their contiguous
    // records (thread g takes entries g, g + G, ...: the paper's coalesced
    // mapping); a thread's few terms sum in FP32
    if (a.fp32 && a.n_p32 > 0) {
        for (int e = gtid; e < a.n_p32; e += gthreads) {
            const float *r = a.rec32 + a.p32_off + (size_t)e * rec32_stride(0);
            const float4 r0 = reinterpret_cast<const float4 *>(r)[0];
            const float4 r1 = reinterpret_cast<const float4 *>(r)[1];
            const float qh = r[rec32_m(0)], ql = r1.w;
#pragma unroll
            for (int q = 0; q < kSmallChunk; ++q) {
                if (q >= nq)
                    break;
                const float dx = (r0.x - s_ph[q][0]) + (r1.x - s_pl[q][0]);
                const float dy = (r0.y - s_ph[q][1]) + (r1.y - s_pl[q][1]);
                const float dz = (r0.z - s_ph[q][2]) + (r1.z - s_pl[q][2]);
                const float rs = esp_rsqrt(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
                acc32[q] += fmaf(qh, rs, ql * rs);
            }
        }
    }
    // every other tile (FP64 points, distributions; FP32 points under FP64),
    // dealt round-robin to the CTAs, one entry per thread
    if (has64) {
        for (int t = blockIdx.x; t < a.n_tiles; t += gridDim.x) {
            const TileMeta m = a.tiles[t];
            if (m.cls == kClassPoint32 && a.fp32)
                continue;
            const bool pts = is_point_class(m.cls);
            const int st = pts ? kPointStride64 : rec64_stride(m.cls & 7);
            for (int j = threadIdx.x; j < m.n; j += kSmallThreads) {
                const double *r = a.rec64 + m.off64 + (size_t)j * st;
#pragma unroll
                for (int q = 0; q < kSmallChunk; ++q) {
                    if (q >= nq)
                        break;
                        if (pts) {
                        const double dx = r[0] - s_pos[q][0], dy = r[1] - s_pos[q][1], dz = r[2] - s_pos[q][2];
                        acc[q] += r[3] * esp_rsqrt(dx * dx + dy * dy + dz * dz);
                    } else {
                        acc[q] += tile_f64_one_any(m.cls, r, 1, s_pos[q][0], s_pos[q][1], s_pos[q][2],
                                                   a.boys64);
                    }
                }
            }
        }
    }
    // fixed-order reduction per position: the FP32 sums as (sum,
    // compensation) pairs by warp shuffles, the FP64 sums (only where this
    // CTA has any) likewise in FP64, then the warps in order in FP64
#pragma unroll
    for (int q = 0; q < kSmallChunk; ++q) {
        if (q >= nq)
            break;
        float sv = acc32[q], cv = 0.0f;
        for (int o = 16; o; o >>= 1) {
            const float so = __shfl_xor_sync(0xffffffffu, sv, o), co = __shfl_xor_sync(0xffffffffu, cv, o);
            two_sum_pair(sv, cv, so, co);
        }
        double v = 0.0;
        if (has64) {
            v = acc[q];
            for (int o = 16; o; o >>= 1)
                v += __shfl_xor_sync(0xffffffffu, v, o);
        }
        if (lane == 0) {
            s_red32[warp][q][0] = sv;
            s_red32[warp][q][1] = cv;
            s_red64[warp][q] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x < nq) {
        double v = 0.0;
        for (int w = 0; w < kSmallThreads / 32; ++w)
            v += (double(s_red32[w][threadIdx.x][0]) + double(s_red32[w][threadIdx.x][1])) +
                 s_red64[w][threadIdx.x];
        a.partial[(size_t)blockIdx.x * n + q0 + threadIdx.x] = v;
    }
}

// ---------------------------------------------------------------------------
// reductions
// ---------------------------------------------------------------------------
// Many partials for few positions: one CTA per position, strided TwoSum per
// thread, then a fixed-order tree over the threads' (sum, compensation) pairs.
constexpr int kWideThreads = 256;

__global__ void __launch_bounds__(kWideThreads) reduce_wide_kernel(const double *__restrict__ partial, int n_splits,
                                                                    int n, double *__restrict__ V)
{
    __shared__ double s_s[kWideThreads], s_c[kWideThreads];
    const int q = blockIdx.x, t = threadIdx.x;
    double sum = 0.0, cmp = 0.0;
    for (int k = t; k < n_splits; k += kWideThreads)
        two_sum_acc(sum, cmp, partial[(size_t)k * n + q]);
    s_s[t] = sum;
    s_c[t] = cmp;
    __syncthreads();
    for (int o = kWideThreads / 2; o > 0; o >>= 1) {
        if (t < o) {
            double a = s_s[t], c = s_c[t] + s_c[t + o];
            two_sum_acc(a, c, s_s[t + o]);
            s_s[t] = a;
            s_c[t] = c;
        }
        __syncthreads();
    }
    if (t == 0)
        V[q] = s_s[0] + s_c[0];
}

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

// one warp per walker: its lanes' electrons by TwoSum, then the lanes in a fixed order
__global__ void walker_kernel(const double *__restrict__ V, int n_walkers, int n_elec, double *__restrict__ E)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
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

cudaError_t launch_batch(int precision, const BatchHeader *hdr, const SysDesc *sys, int max_sys, int *counter,
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
        e = launch_batch_shape<NT, PPT, PR>(hdr, sys, counter, max_items, boys32, boys64, boysdd, tile_cap, num_sms, smem, \
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

// Slices of the environment's entries: about 8 CTAs per SM over all chunks of
// positions, so that with more positions each thread takes more entries and
// the per-position reduction is amortised over more terms.
int small_n_splits(int n_tiles, int num_sms, int n)
{
    const int chunks = std::max(1, (n + kSmallChunk - 1) / kSmallChunk);
    return std::max(1, std::min(n_tiles, 8 * num_sms / chunks));
}

cudaError_t launch_small_n(const SmallArgs &a, int n_splits, double *V, cudaStream_t s)
{
    if (a.n_pos <= 0 || a.n_pos > kSmallN)
        return cudaErrorInvalidValue;
    const dim3 grid(n_splits, (a.n_pos + kSmallChunk - 1) / kSmallChunk);
    small_n_kernel<<<grid, kSmallThreads, 0, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return e;
    reduce_wide_kernel<<<a.n_pos, kWideThreads, 0, s>>>(a.partial, n_splits, a.n_pos, V);
    return cudaGetLastError();
}

cudaError_t launch_reduce(const double *partial, int n_splits, int n, double *V, cudaStream_t s, const int *perm)
{
    if (n <= 0)
        return cudaSuccess;
    const int grid = (n + 31) / 32;
    // more slices where the partials are many and the positions few
    if (n_splits > 64)
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
