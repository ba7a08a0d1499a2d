// The parts of an FP32C evaluation that need FP64 accuracy, in pairs of FP32
// numbers (esp_dd.h): every point charge of FP64 tiles at every position, and
// the near (position, tile) blocks, which the FP32C kernel leaves out.
//
// One position per thread, 128 per CTA; a CTA stages one tile's dd records in
// shared memory and all its threads read them as broadcasts, two records per
// packed FP32 operation.  Bound by the FP32 pipe: 75 operations per two charges,
// about 130 per two s-distributions with their Boys values.  In FP64 (1/63 of
// the rate) the same blocks took 500 of the 650 us of 10,000 positions x 2,200
// entries whose tiles' spheres cover the QM region; here they take 53.
#include "esp_ddsum.cuh"

#include <algorithm>

namespace esp {

namespace {

constexpr int kDdThreads = 128;
constexpr int kDdWordsMax = dd_far_words(kDdGeneralMaxL) + dd_gen_words(kDdGeneralMaxL); // the largest tile staged

__global__ void __launch_bounds__(kDdThreads, 4) dd_sum_kernel(EvalArgs a, const int *__restrict__ list, int n_list)
{
    extern __shared__ float4 smem4[];
    const float *s_rec = reinterpret_cast<const float *>(smem4);
    const int i = blockIdx.x * kDdThreads + threadIdx.x, ic = min(i, a.n_pos - 1);
    const DdPos c = dd_position(a.pos, ic);
    const bool in_range = dd_in_range(c.h, a.dd_lim);
    double acc = 0.0;
    for (int k = blockIdx.y; k < n_list; k += gridDim.y) {
        const TileMeta m = a.tiles[list[k]];
        const bool pts = m.cls == kClassPoint;
        bool mine = true, f, r;
        if (!pts)
            classify_tile(m, c.h[0], c.h[1], c.h[2], a.near_r, mine, f, r);
        // (also: the previous tile is fully consumed)
        if (!__syncthreads_or(mine))
            continue;
        if (m.offdd < 0 || !(pts || dd_has_general(m))) {
            if (pts) { // (one chain of additions over the tiles)
                const double p[1][3] = {{a.pos.x64[ic], a.pos.y64[ic], a.pos.z64[ic]}};
                double v[1] = {acc};
                tile_points_f64<1>(a.rec64 + m.off64, m.n, p, v);
                acc = v[0];
            } else if (mine) {
                acc += tile_f64_one_any(m.cls, a.rec64 + m.off64, m.n, a.pos.x64[ic], a.pos.y64[ic], a.pos.z64[ic],
                                        a.boys64);
            }
            continue;
        }
        const int n4 = dd_pad(m.n);
        copy_tile(smem4, reinterpret_cast<const float4 *>(a.recdd) + m.offdd, dd_words(m) * n4 / 4);
        __syncthreads();
        if (pts) {
            float r2min;
            double v = dd_sum_points(s_rec, n4, c, &r2min);
            // closer than the dd words resolve, or out of their range
            if (!(r2min >= dd_min_r2(a.dd_lim)) || !in_range)
                v = point_tile_f64(a.rec64 + m.off64, m.n, a.pos.x64[ic], a.pos.y64[ic], a.pos.z64[ic]);
            acc += v;
        } else if (__any_sync(0xffffffffu, mine)) {
            double v = dd_sum_general(m.cls, s_rec, n4, c, a.boysdd);
            if (mine && !in_range)
                v = tile_f64_one_any(m.cls, a.rec64 + m.off64, m.n, a.pos.x64[ic], a.pos.y64[ic], a.pos.z64[ic],
                                     a.boys64);
            acc += mine ? v : 0.0;
        }
    }
    if (i < a.n_pos)
        a.partial[(size_t)blockIdx.y * a.n_pos + i] = acc;
}

// ---------------------------------------------------------------------------
// FP64 evaluations.  Every entry whose Gaussian is negligible at a position
// (T = p |P - C|^2 >= 45 and a margin) takes the far form of esp_dd.h in three
// FP32 words: about 170 packed FP32 operations per two monopoles, 400 with L = 1
// and 750 with L = 2.  (The orders above the monopole in two words were faster,
// 2,048 positions x 48,000 distributions in 1.5 ms, but erred by 7e-15 and more
// of an order that stands alone; in three 2.0 ms and 1e-16.)  The others take the
// FP64 code, each lane its own entries: a warp runs as many as its busiest lane
// has, not as many as any lane has (with two words 1.56 -> 1.52 ms).  Bound by the
// FP64 pipe where exponents are small (those entries: some 40 operations of 64
// cycles), by FP32 otherwise.  All in FP64, 2,048 x 48,000 took 9.5 ms.
// ---------------------------------------------------------------------------
constexpr int kTdWordsMax = dd_far_words(kMaxL);

// The far pairs of a chunk of at most 64 records; near: bits of the records
// that this lane leaves out.  lo: the smallest |P - C|^2 met.
template <int L>
__device__ __noinline__ double td_chunk(const float *__restrict__ s_rec, int n4, int j0, int j1, const DdPos c,
                                        unsigned long long near, float *lo)
{
    const DdTile t = {s_rec, n4};
    double acc = 0.0;
    float r2min = *lo;
    for (int b = j0; b < j1; b += 16) {
        TdSum sum;
        sum.clear();
        const int e = min(j1, b + 16);
#pragma unroll 1
        for (int j = b; j < e; j += 2) {
            const bool u0 = !(near >> (j - j0) & 1), u1 = !(near >> (j - j0 + 1) & 1);
            if (!__any_sync(0xffffffffu, u0 || u1))
                continue;
            f2 r2;
            td_far<L>(t, j, c, u0, u1, sum, r2);
            r2min = fminf(r2min, fminf(r2.x, r2.y));
        }
        acc += sum.total();
    }
    *lo = r2min;
    return acc;
}
__device__ __noinline__ double td_points(const float *__restrict__ s_rec, int n4, const DdPos c, float *lo)
{
    const DdTile t = {s_rec, n4};
    double acc = 0.0;
    float r2min = *lo;
    for (int b = 0; b < n4; b += 16) {
        TdSum sum;
        sum.clear();
        const int e = min(n4, b + 16);
#pragma unroll 1
        for (int j = b; j < e; j += 2) {
            f2 r2;
            td_point(t, j, c, sum, r2);
            r2min = fminf(r2min, fminf(r2.x, r2.y));
        }
        acc += sum.total();
    }
    *lo = r2min;
    return acc;
}
__device__ __noinline__ double near_entry(int cls, const double *__restrict__ r, double x, double y, double z,
                                          const double *__restrict__ boys64)
{
    return tile_f64_one_any(cls, r, 1, x, y, z, boys64);
}

__global__ void __launch_bounds__(kDdThreads, 4) potential_td_kernel(EvalArgs a)
{
    extern __shared__ float4 smem4[];
    const float *s_rec = reinterpret_cast<const float *>(smem4);
    const int i = blockIdx.x * kDdThreads + threadIdx.x, ic = min(i, a.n_pos - 1);
    const DdPos c = dd_position(a.pos, ic);
    const double x = a.pos.x64[ic], y = a.pos.y64[ic], z = a.pos.z64[ic];
    const bool in_range = dd_in_range(c.h, a.dd_lim);
    const float min_r2 = td_min_r2(a.dd_lim);
    double S = 0.0, Cc = 0.0;
    const int shift = a.grp_shift[0], part = a.tile_size >> shift;
    for (int k = blockIdx.y; k < a.n_tiles << shift; k += gridDim.y) {
        const TileMeta m = a.tiles[k >> shift];
        const bool pts = is_point_class(m.cls);
        // this part's records [p0, p0 + n)
        const int p0 = (k & ((1 << shift) - 1)) * part, n = min(m.n - p0, part);
        if (n <= 0)
            continue;
        const double *rec64 = a.rec64 + m.off64 + (size_t)p0 * (pts ? kPointStride64 : rec64_stride(m.cls & 7));
        if (m.offdd < 0) {
            two_sum_acc(S, Cc, pts ? point_tile_f64(rec64, n, x, y, z)
                                   : tile_f64_one_any(m.cls, rec64, n, x, y, z, a.boys64));
            continue;
        }
        const int n4 = dd_pad(n), L = m.cls & 7;
        __syncthreads(); // the previous tile is fully consumed
        copy_part(smem4, reinterpret_cast<const float4 *>(a.recdd) + m.offdd, pts ? kDdPointWords : dd_far_words(L),
                  dd_pad(m.n), p0, n4);
        __syncthreads();
        float r2min = 1.0f;
        double v = 0.0;
        if (pts) {
            v = td_points(s_rec, n4, c, &r2min);
        } else {
            const float ex = c.h[0] - m.cx, ey = c.h[1] - m.cy, ez = c.h[2] - m.cz;
            const float d = sqrtf(ex * ex + ey * ey + ez * ez) - m.rad;
            const bool far = __all_sync(0xffffffffu, d > 0.0f && td_is_far(m.pmin * d * d, d * d, min_r2));
            const DdTile t = {s_rec, n4};
            for (int j0 = 0; j0 < n4; j0 += 64) {
                const int j1 = min(n4, j0 + 64);
                unsigned long long near = 0ull;
                if (!far) { // which records are near this lane's position
                    for (int j = j0; j < j1; j += 2) {
                        const f2 dx = t(0, j) - f2(c.h[0]), dy = t(1, j) - f2(c.h[1]), dz = t(2, j) - f2(c.h[2]);
                        const f2 r2 = esp_fma(dx, dx, esp_fma(dy, dy, dz * dz)), T = t(10, j) * r2;
                        near |= (unsigned long long)((td_is_far(T.x, r2.x, min_r2) ? 0u : 1u) |
                                                     (td_is_far(T.y, r2.y, min_r2) ? 0u : 2u))
                                << (j - j0);
                    }
                }
                switch (L) {
                case 0: v += td_chunk<0>(s_rec, n4, j0, j1, c, near, &r2min); break;
                case 1: v += td_chunk<1>(s_rec, n4, j0, j1, c, near, &r2min); break;
                case 2: v += td_chunk<2>(s_rec, n4, j0, j1, c, near, &r2min); break;
                case 3: v += td_chunk<3>(s_rec, n4, j0, j1, c, near, &r2min); break;
                default: v += td_chunk<4>(s_rec, n4, j0, j1, c, near, &r2min); break;
                }
                if (n - j0 < 64) // (padding repeats the last record)
                    near &= (1ull << (n - j0)) - 1ull;
                for (; near; near &= near - 1)
                    v += near_entry(m.cls, rec64 + (size_t)(j0 + __ffsll((long long)near) - 1) * rec64_stride(L), x, y,
                                    z, a.boys64);
            }
        }
        // closer than the words resolve, or out of their range
        if (!(r2min >= min_r2) || !in_range)
            v = pts ? point_tile_f64(rec64, n, x, y, z) : tile_f64_one_any(m.cls, rec64, n, x, y, z, a.boys64);
        two_sum_acc(S, Cc, v);
    }
    if (i < a.n_pos)
        a.partial[(size_t)blockIdx.y * a.n_pos + i] = S + Cc;
}

// dd records of one tile per CTA; the padding repeats the last record's
// coordinates with zero coefficients
__global__ void dd_build_kernel(const TileMeta *__restrict__ tiles, const double *__restrict__ rec64, double q,
                                float *__restrict__ recdd)
{
    const TileMeta m = tiles[blockIdx.x];
    if (m.offdd < 0)
        return;
    const bool pts = is_point_class(m.cls);
    const int n4 = dd_pad(m.n), st = pts ? kPointStride64 : rec64_stride(m.cls & 7);
    float *out = recdd + (size_t)m.offdd * 4;
    for (int j = threadIdx.x; j < n4; j += blockDim.x) {
        dd_convert(m, rec64 + m.off64 + (size_t)min(j, m.n - 1) * st, q, out + j, n4);
        if (j >= m.n)
            dd_zero_coefficients(m, out + j, n4);
    }
}

} // namespace

int dd_sum_splits(int n, int n_list, int num_sms)
{
    if (n_list <= 0)
        return 0;
    const int blocks = (n + kDdThreads - 1) / kDdThreads;
    return std::max(1, std::min(n_list, (8 * num_sms + blocks - 1) / blocks));
}

cudaError_t launch_dd_sum(const EvalArgs &a, const int *list, int n_list, int n_splits, cudaStream_t s)
{
    if (a.n_pos <= 0 || n_list <= 0)
        return cudaSuccess;
    const size_t smem = (size_t)a.tile_size * kDdWordsMax * sizeof(float);
    cudaError_t e = allow_smem(dd_sum_kernel, (size_t)kMaxTileSize * kDdWordsMax * sizeof(float));
    if (e != cudaSuccess)
        return e;
    const dim3 grid((a.n_pos + kDdThreads - 1) / kDdThreads, n_splits);
    dd_sum_kernel<<<grid, kDdThreads, smem, s>>>(a, list, n_list);
    return cudaGetLastError();
}

int td_splits(int n, int n_tiles, int num_sms, int &shift)
{
    const int blocks = (n + kDdThreads - 1) / kDdThreads;
    // One wave of the four CTAs an SM holds, two where that would leave fewer
    // than 16 splits: a partial second wave costs a whole one (2,048 positions x
    // 889 tiles: 38 splits, one wave, 1.56 ms; 47: 2.20; 57: 1.74; 76: 1.71).
    const int wave = 4 * num_sms / blocks;
    const int want = std::max(1, wave >= 16 ? wave : 8 * num_sms / blocks);
    // parts of tiles until a split has eight of them (1,999 positions x 39 tiles:
    // 188 us in whole tiles, 151 in quarters, 160 in eighths)
    shift = 0;
    while (shift < kMaxPartShift && n_tiles << shift < 8 * want)
        ++shift;
    return std::max(1, std::min(n_tiles << shift, want));
}

cudaError_t launch_td(const EvalArgs &a, cudaStream_t s)
{
    if (a.n_pos <= 0)
        return cudaSuccess;
    const size_t smem = (size_t)a.tile_size * kTdWordsMax * sizeof(float);
    cudaError_t e = allow_smem(potential_td_kernel, (size_t)kMaxTileSize * kTdWordsMax * sizeof(float));
    if (e != cudaSuccess)
        return e;
    const dim3 grid((a.n_pos + kDdThreads - 1) / kDdThreads, a.n_splits);
    potential_td_kernel<<<grid, kDdThreads, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_dd_build(const TileMeta *tiles, int n_tiles, const double *rec64, double q, float *recdd,
                            cudaStream_t s)
{
    if (n_tiles <= 0)
        return cudaSuccess;
    dd_build_kernel<<<n_tiles, 64, 0, s>>>(tiles, rec64, q, recdd);
    return cudaGetLastError();
}

} // namespace esp
