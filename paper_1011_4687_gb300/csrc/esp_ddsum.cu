// The parts of an FP32C evaluation that need FP64 accuracy, in pairs of FP32
// numbers (esp_dd.h): every point charge of FP64 tiles at every position, and
// the near (position, tile) blocks, which the FP32C kernel leaves out.
//
// One position per thread, 128 per CTA; a CTA stages one tile's dd records in
// shared memory and all its threads read them as broadcasts, two records per
// packed FP32 operation.  Bound by the FP32 pipe: 75 operations per two charges,
// about 130 per two s-distributions with their Boys values.  In FP64 (1/63 of
// the rate) the same blocks took 500 of the 650 us of 10,000 positions x 2,200
// entries whose tiles' spheres cover the QM region.
#include "esp_ddsum.cuh"

#include <algorithm>

namespace esp {

namespace {

constexpr int kDdThreads = 128;
constexpr int kDdWordsMax = dd_words(kDdGeneralMaxL); // the largest tile staged here

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
        if (m.offdd < 0) {
            if (mine)
                acc += pts ? point_tile_f64(a.rec64 + m.off64, m.n, a.pos.x64[ic], a.pos.y64[ic], a.pos.z64[ic])
                           : tile_f64_one_any(m.cls, a.rec64 + m.off64, m.n, a.pos.x64[ic], a.pos.y64[ic],
                                              a.pos.z64[ic], a.boys64);
            continue;
        }
        const int n4 = dd_pad(m.n);
        copy_tile(smem4, reinterpret_cast<const float4 *>(a.recdd) + m.offdd, dd_words(m.cls) * n4 / 4);
        __syncthreads();
        if (pts) {
            float r2min;
            double v = dd_sum_points(s_rec, n4, c, &r2min);
            // closer than the dd words resolve, or out of their range
            if (!(r2min >= kDdMinR2) || !in_range)
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
        dd_convert(m.cls, rec64 + m.off64 + (size_t)min(j, m.n - 1) * st, q, out + j, n4);
        if (j >= m.n)
            dd_zero_coefficients(m.cls, out + j, n4);
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
    cudaError_t e = cudaFuncSetAttribute(dd_sum_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess)
        return e;
    const dim3 grid((a.n_pos + kDdThreads - 1) / kDdThreads, n_splits);
    dd_sum_kernel<<<grid, kDdThreads, smem, s>>>(a, list, n_list);
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
