// Device code shared by the kernels that sum tiles in pairs of FP32 numbers
// (esp_dd.h): tile staging, the words of a position, a tile's sum at one
// position.
#pragma once

#include "esp_dd.h"
#include "esp_eval_core.h"
#include "esp_kernels.h"

namespace esp {

namespace {

__device__ __forceinline__ void copy_tile(float4 *__restrict__ dst, const float4 *__restrict__ src, int nvec)
{
    for (int i = threadIdx.x; i < nvec; i += blockDim.x)
        dst[i] = __ldg(src + i);
}

// words [0, words) of records [j0, j0 + n4p) of a dd tile of n4 records (j0 and
// n4p multiples of 4), as a tile of n4p records
__device__ __forceinline__ void copy_part(float4 *__restrict__ dst, const float4 *__restrict__ src, int words, int n4,
                                          int j0, int n4p)
{
    if (n4p == n4)
        return copy_tile(dst, src, words * n4 / 4);
    const int q = n4p / 4;
    for (int i = threadIdx.x; i < words * q; i += blockDim.x) {
        const int w = i / q;
        dst[i] = __ldg(src + w * (n4 / 4) + j0 / 4 + (i - w * q));
    }
}

__device__ __forceinline__ DdPos dd_position(const Staged &p, int i)
{
    return {{p.xh[i], p.yh[i], p.zh[i]}, {p.xm[i], p.ym[i], p.zm[i]}, {p.xr[i], p.yr[i], p.zr[i]}};
}

// the position's hi words allow exact offsets (false for NaN)
__device__ __forceinline__ bool dd_in_range(const float (&h)[3], float lim)
{
    return fabsf(h[0]) <= lim && fabsf(h[1]) <= lim && fabsf(h[2]) <= lim;
}

__device__ __forceinline__ double dd_total(const dd &s)
{
    return ((double)s.h.x + (double)s.h.y) + (double)(s.l.x + s.l.y);
}

// Staged dd point tile at one position; r2min: the smallest squared distance.
// Bound by the FP32 pipe (about 75 packed operations per two charges) instead
// of the FP64 pipe, whose 1/63 rate made 200 nuclei cost more than 2,000
// s-charges in FP32.
__device__ __forceinline__ double dd_sum_points(const float *__restrict__ s_rec, int n4, const DdPos &c, float *r2min)
{
    const DdTile t = {s_rec, n4};
    dd acc = {f2(0.0f), f2(0.0f)};
    float lo = 3.0e38f;
#pragma unroll 2
    for (int j = 0; j < n4; j += 2) {
        f2 r2;
        acc = dd_add(acc, dd_point(t, j, c, r2));
        lo = fminf(lo, fminf(r2.x, r2.y));
    }
    *r2min = lo;
    return dd_total(acc);
}

// Staged dd distribution tile (class L <= 2, not short-range) at one position.
template <int L>
__device__ __forceinline__ double dd_sum_general_one(const float *__restrict__ s_rec, int n4, const DdPos &c,
                                                     const float *__restrict__ boysdd)
{
    const DdTile t = {s_rec, n4};
    dd acc = {f2(0.0f), f2(0.0f)};
#pragma unroll 1
    for (int j = 0; j < n4; j += 2)
        acc = dd_add(acc, dd_general<L>(t, j, c, dd_far_words(L), boysdd));
    return dd_total(acc);
}
__device__ __forceinline__ double dd_sum_general(int L, const float *__restrict__ s_rec, int n4, const DdPos &c,
                                                 const float *__restrict__ boysdd)
{
    return L == 0   ? dd_sum_general_one<0>(s_rec, n4, c, boysdd)
           : L == 1 ? dd_sum_general_one<1>(s_rec, n4, c, boysdd)
                    : dd_sum_general_one<2>(s_rec, n4, c, boysdd);
}

__device__ __forceinline__ double point_tile_f64(const double *__restrict__ pts, int n, double x, double y, double z)
{
    const double c[1][3] = {{x, y, z}};
    double v[1] = {0.0};
    tile_points_f64<1>(pts, n, c, v);
    return v[0];
}

} // namespace

} // namespace esp
