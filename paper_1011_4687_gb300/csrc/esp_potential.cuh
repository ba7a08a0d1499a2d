// Potential kernel templates (FP32C, FP64, batched persistent) for sm_103a.
//
// The paper's kernel (Sec. III, Eq. blockSum and Eq. coalease) splits the cell
// sum over N_B blocks of N_th threads, each thread striding through the cell
// array so that neighbouring threads read neighbouring cells (coalescing), and
// reduces per block in shared memory; one position r_new sits in constant
// memory.  Here many positions are evaluated per launch, so the roles turn
// around: each thread keeps PPT positions in registers, a CTA stages one tile
// of distributions at a time in shared memory with coalesced 16-byte loads,
// and every warp reads the tile's records as same-address broadcasts.  Tiles
// are dealt round-robin to `n_splits` CTAs per position block; each split
// writes its own partial, and a separate kernel sums the partials in a
// fixed order (deterministic, no atomics on the result).
//
// Only esp_shape.cu instantiates these templates, once per launch shape and
// object file (the shape lists are in esp_shapes.h), so that the shapes
// compile in parallel.
#pragma once

#include "esp_ddsum.cuh"
#include "esp_eval_core.h"
#include "esp_kernels.h"

namespace esp {

namespace {

// The dd sums as calls (the batched kernel keeps its registers for the FP32 sums).
__device__ __noinline__ double dd_points_call(const float *__restrict__ s_rec, int n4, const DdPos c, float *r2min)
{
    return dd_sum_points(s_rec, n4, c, r2min);
}
__device__ __noinline__ double dd_general_call(int L, const float *__restrict__ s_rec, int n4, const DdPos c,
                                               const float *__restrict__ boysdd)
{
    return dd_sum_general(L, s_rec, n4, c, boysdd);
}

// ---------------------------------------------------------------------------
// FP32C kernel
// ---------------------------------------------------------------------------
// One CTA's work in the FP32C kernel: position block bx against the tiles of
// split `split` (tiles split, split + n_splits, ...).  The Boys table is
// already in shared memory (s_boys); s_tile4 holds one staged tile, s_acc one
// FP64 sum per position (ALL).
// ALL: also the FP64 point charges and the near blocks (the batched kernel);
// otherwise the dd kernel (esp_ddsum.cu) sums those and this one only leaves
// them out: their code and its calls cost the far form's loops registers
// (65,536 positions x 109,368 distributions: 9.48 ms with, 9.1 ms without).
template <int NT, int PPT, bool ALL>
__device__ __forceinline__ void cta_f32c(const EvalArgs &a, int bx, int split, float4 *s_tile4,
                                         const float *s_boys, double *s_acc)
{
    const int base = bx * NT * PPT + threadIdx.x;
    // The FP32 sums and the positions' words live in registers from tile to
    // tile; the FP64 sums, which few tiles add to, stay in shared memory.  (The
    // words from L1 again for each tile gave the far form's loops 24 registers
    // and no spills, but cost more than they gave: the records stream through
    // the same L1.  65,536 positions x 19.7 million distributions 1,297 ms
    // against 1,274, 131,072 x 1.1 million 160.9 against 158.6.)
    auto pos_of = [&](int q) { return min(base + q * NT, a.n_pos - 1); };
    double *acc64 = s_acc + threadIdx.x; // [q * NT]
    float S[PPT], Cc[PPT];
#pragma unroll
    for (int q = 0; q < PPT; ++q) {
        S[q] = 0.0f;
        Cc[q] = 0.0f;
        if (ALL)
            acc64[q * NT] = 0.0;
    }
    // the sums of position pairs (used when PPT is even)
    constexpr int NP = PPT / 2 > 0 ? PPT / 2 : 1;
    f2 S2[NP], C2[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        S2[q] = f2(0.0f);
        C2[q] = f2(0.0f);
    }
    float ch[PPT][3], cl[PPT][3];
#pragma unroll
    for (int q = 0; q < PPT; ++q) {
        const int ic = pos_of(q);
        ch[q][0] = a.pos.xh[ic];
        ch[q][1] = a.pos.yh[ic];
        ch[q][2] = a.pos.zh[ic];
        cl[q][0] = a.pos.xl[ic];
        cl[q][1] = a.pos.yl[ic];
        cl[q][2] = a.pos.zl[ic];
    }
    // the same positions as lane pairs
    f2 ch2[NP][3], cl2[NP][3];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const int q0 = 2 * q < PPT ? 2 * q : 0, q1 = 2 * q + 1 < PPT ? 2 * q + 1 : 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            ch2[q][d] = f2(ch[q0][d], ch[q1][d]);
            cl2[q][d] = f2(cl[q0][d], cl[q1][d]);
        }
    }
    const float near_r = a.near_r;
    // this split's group and its place among the group's splits
    int g = 0;
    while (g + 1 < a.n_groups && split >= a.grp_split[g + 1])
        ++g;
    const int g_stride = a.grp_split[g + 1] - a.grp_split[g];
    const int shift = ALL ? 0 : a.grp_shift[g];
    const int g_units = (a.grp_tile[g + 1] - a.grp_tile[g]) << shift;
    for (int u = split - a.grp_split[g]; u < g_units; u += g_stride) {
        const TileMeta m = a.tiles[a.grp_tile[g] + (u >> shift)];
        // this part's records [j0, j0 + n)
        const int j0 = ALL ? 0 : (u & ((1 << shift) - 1)) * (a.tile_size >> shift);
        const int n = ALL ? m.n : min(m.n - j0, a.tile_size >> shift);
        if (!ALL && n <= 0)
            continue;
        if (!ALL && m.cls == kClassPoint)
            continue;
        __syncthreads(); // previous tile fully consumed
        const bool pts = ALL && m.cls == kClassPoint;
        const bool ddt = a.recdd && m.offdd >= 0;
        const int n4 = dd_pad(m.n);
        const float4 *s_dd = reinterpret_cast<const float4 *>(a.recdd) + (ddt ? m.offdd : 0);
        const float4 *src = pts ? (ddt ? s_dd : reinterpret_cast<const float4 *>(a.rec64 + m.off64))
                                : reinterpret_cast<const float4 *>(a.rec32 + m.off32 + j0 * rec32_stride_cls(m.cls));
        const int nvec = pts ? (ddt ? kDdPointWords * n4 / 4 : m.n * 2)
                             : (n * rec32_stride_cls(m.cls)) / 4;
        copy_tile(s_tile4, src, nvec);
        if (!ALL)
            asm volatile("cp.async.wait_all;" ::: "memory"); // the Boys table, once
        __syncthreads();
        if (m.cls == kClassPoint32) {
            // small point charges: the far form of an L = 0 record, no near path
            const float *s_rec = reinterpret_cast<const float *>(s_tile4);
            // (absolute hi words: th = 0 - C_hi, the exact offset form)
            if constexpr (PPT % 2 == 0) {
                f2 wq[NP], th2[NP][3];
#pragma unroll
                for (int q = 0; q < NP; ++q)
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        th2[q][d] = f2(0.0f) - ch2[q][d];
                tile_f32c2<0, NP, true, false, false>(s_rec, n, th2, cl2, cl2, wq, S2, C2, s_boys);
            } else {
                bool none[PPT];
                float th[PPT][3];
#pragma unroll
                for (int q = 0; q < PPT; ++q) {
                    none[q] = false;
#pragma unroll
                    for (int d = 0; d < 3; ++d)
                        th[q][d] = 0.0f - ch[q][d];
                }
                tile_f32c<0, PPT, true, false, false>(s_rec, n, th, cl, cl, none, S, Cc, s_boys);
            }
            continue;
        }
        if (ALL && pts && !ddt) {
            double c64[PPT][3], v[PPT];
#pragma unroll
            for (int q = 0; q < PPT; ++q) {
                const int ic = pos_of(q);
                c64[q][0] = a.pos.x64[ic];
                c64[q][1] = a.pos.y64[ic];
                c64[q][2] = a.pos.z64[ic];
                v[q] = acc64[q * NT];
            }
            tile_points_f64<PPT>(reinterpret_cast<const double *>(s_tile4), m.n, c64, v);
#pragma unroll
            for (int q = 0; q < PPT; ++q)
                acc64[q * NT] = v[q];
            continue;
        }
        if (ALL && pts) {
#pragma unroll 1
            for (int q = 0; q < PPT; ++q) {
                const int ic = pos_of(q);
                const DdPos c = dd_position(a.pos, ic);
                float r2min;
                double v = dd_points_call(reinterpret_cast<const float *>(s_tile4), n4, c, &r2min);
                // closer than the dd words resolve, or out of their range
                if (!(r2min >= dd_min_r2(a.dd_lim)) || !dd_in_range(c.h, a.dd_lim))
                    v = point_tile_f64(a.rec64 + m.off64, m.n, a.pos.x64[ic], a.pos.y64[ic], a.pos.z64[ic]);
                acc64[q * NT] += v;
            }
            continue;
        }
        bool nearq[PPT];
        bool any_near = false, lane_far = true, lane_rel = true;
#pragma unroll
        for (int q = 0; q < PPT; ++q) {
            bool f, r;
            classify_tile(m, ch[q][0], ch[q][1], ch[q][2], near_r, nearq[q], f, r);
            any_near |= nearq[q];
            lane_far &= f;
            lane_rel &= r;
        }
        const bool far = __all_sync(0xffffffffu, lane_far);
        const bool rel = __all_sync(0xffffffffu, lane_rel); // implies far
        const bool sel = __any_sync(0xffffffffu, any_near); // warp-uniform: any term to select away
        const float *s_rec = reinterpret_cast<const float *>(s_tile4);
        const float ct[3] = {m.cx, m.cy, m.cz}; // the records' reference point T
        if constexpr (PPT % 2 == 0) {
            // two positions per packed FP32 instruction
            f2 wq[NP], th2[NP][3], dq2[NP][3];
#pragma unroll
            for (int q = 0; q < NP; ++q) {
                wq[q] = f2(nearq[2 * q] ? 0.0f : 1.0f, nearq[2 * q + 1] ? 0.0f : 1.0f);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    th2[q][d] = f2(ct[d]) - ch2[q][d];
                    dq2[q][d] = th2[q][d] - cl2[q][d];
                }
            }
#define ESP_TILE(CLS, LL, SH)                                                                         \
    case CLS:                                                                                         \
        if (rel && !sel)                                                                              \
            tile_f32c2<LL, NP, true, SH, false, true>(s_rec, n, th2, cl2, dq2, wq, S2, C2, s_boys); \
        else if (far && !sel)                                                                         \
            tile_f32c2<LL, NP, true, SH, false>(s_rec, n, th2, cl2, dq2, wq, S2, C2, s_boys);       \
        else if (far)                                                                                 \
            tile_f32c2<LL, NP, true, SH, true>(s_rec, n, th2, cl2, dq2, wq, S2, C2, s_boys);        \
        else                                                                                          \
            tile_f32c2<LL, NP, false, SH, true>(s_rec, n, th2, cl2, dq2, wq, S2, C2, s_boys);       \
        break;
            switch (m.cls) {
                ESP_TILE(0, 0, false)
                ESP_TILE(1, 1, false)
                ESP_TILE(2, 2, false)
                ESP_TILE(3, 3, false)
                ESP_TILE(4, 4, false)
                ESP_TILE(8, 0, true)
                ESP_TILE(9, 1, true)
                ESP_TILE(10, 2, true)
                ESP_TILE(11, 3, true)
                default:
                ESP_TILE(12, 4, true)
            }
#undef ESP_TILE
        } else {
            float th[PPT][3], dq[PPT][3];
#pragma unroll
            for (int q = 0; q < PPT; ++q)
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    th[q][d] = ct[d] - ch[q][d];
                    dq[q][d] = th[q][d] - cl[q][d];
                }
#define ESP_TILE(CLS, LL, SH)                                                                         \
    case CLS:                                                                                         \
        if (rel && !sel)                                                                              \
            tile_f32c<LL, PPT, true, SH, false, true>(s_rec, n, th, cl, dq, nearq, S, Cc, s_boys);  \
        else if (far && !sel)                                                                         \
            tile_f32c<LL, PPT, true, SH, false>(s_rec, n, th, cl, dq, nearq, S, Cc, s_boys);        \
        else if (far)                                                                                 \
            tile_f32c<LL, PPT, true, SH, true>(s_rec, n, th, cl, dq, nearq, S, Cc, s_boys);         \
        else                                                                                          \
            tile_f32c<LL, PPT, false, SH, true>(s_rec, n, th, cl, dq, nearq, S, Cc, s_boys);        \
        break;
            switch (m.cls) {
                ESP_TILE(0, 0, false)
                ESP_TILE(1, 1, false)
                ESP_TILE(2, 2, false)
                ESP_TILE(3, 3, false)
                ESP_TILE(4, 4, false)
                ESP_TILE(8, 0, true)
                ESP_TILE(9, 1, true)
                ESP_TILE(10, 2, true)
                ESP_TILE(11, 3, true)
                default:
                ESP_TILE(12, 4, true)
            }
#undef ESP_TILE
        }
        if (!ALL || m.vmax < kNearVmax || !(near_r > 0.0f))
            continue; // (block-uniform) no position can be near
        if (ddt && dd_has_general(m)) {
            // the CTA stages the tile's dd records; a warp with a near lane
            // sums them at its positions
            if (!__syncthreads_or(any_near))
                continue;
            copy_tile(s_tile4, s_dd, dd_words(m) * n4 / 4);
            __syncthreads();
            const float *s_rec_dd = reinterpret_cast<const float *>(s_tile4);
#pragma unroll
            for (int q = 0; q < PPT; ++q) {
                if (!__any_sync(0xffffffffu, nearq[q]))
                    continue;
                const int ic = pos_of(q);
                const DdPos c = dd_position(a.pos, ic);
                double v = dd_general_call(m.cls, s_rec_dd, n4, c, a.boysdd);
                if (nearq[q] && !dd_in_range(c.h, a.dd_lim))
                    v = tile_f64_one_any(m.cls, a.rec64 + m.off64, m.n, a.pos.x64[ic], a.pos.y64[ic], a.pos.z64[ic],
                                         a.boys64);
                if (nearq[q])
                    acc64[q * NT] += v;
            }
        } else if (any_near) {
#pragma unroll
            for (int q = 0; q < PPT; ++q) {
                if (nearq[q]) {
                    const int ic = pos_of(q);
                    acc64[q * NT] += tile_f64_one_any(m.cls, a.rec64 + m.off64, m.n, a.pos.x64[ic], a.pos.y64[ic],
                                                      a.pos.z64[ic], a.boys64);
                }
            }
        }
    }
    if (!ALL) // (a split without a part)
        asm volatile("cp.async.wait_all;" ::: "memory");
    if constexpr (PPT % 2 == 0) {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            S[2 * q] = S2[q].x;
            S[2 * q + 1] = S2[q].y;
            Cc[2 * q] = C2[q].x;
            Cc[2 * q + 1] = C2[q].y;
        }
    }
#pragma unroll
    for (int q = 0; q < PPT; ++q) {
        const int i = base + q * NT;
        if (!ALL && a.pairs) {
            if (i < a.n_pos)
                reinterpret_cast<float2 *>(a.partial)[(size_t)split * a.n_pos + i] = make_float2(S[q], Cc[q]);
        } else if (i < a.n_pos)
            a.partial[(size_t)split * a.n_pos + i] = ((double)S[q] + (double)Cc[q]) + (ALL ? acc64[q * NT] : 0.0);
    }
}

template <int NT, int PPT>
__global__ void __launch_bounds__(NT, 512 / NT) potential_f32c_kernel(EvalArgs a)
{
    extern __shared__ float4 smem4[];
    float4 *s_tile4 = smem4;
    float *s_boys = reinterpret_cast<float *>(smem4 + (a.tile_size * kRec32MaxStride) / 4);
    // The Boys table comes in asynchronously beside the first tile (a CTA of a
    // short call has one or two tiles; the copy through registers took a fifth
    // of its time); the loop's first barrier follows the wait.
    constexpr int nb = kBoys32Rows * kBoys32Row;
    const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(s_boys));
    for (int i = threadIdx.x; i < nb / 4; i += NT)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * i), "l"(a.boys32 + 4 * i) : "memory");
    if (threadIdx.x < nb % 4)
        s_boys[nb - 1 - threadIdx.x] = a.boys32[nb - 1 - threadIdx.x];
    cta_f32c<NT, PPT, false>(a, blockIdx.x, blockIdx.y, s_tile4, s_boys, nullptr);
    asm volatile("cp.async.wait_all;" ::: "memory"); // (a CTA without tiles)
}

// ---------------------------------------------------------------------------
// FP64 kernel
// ---------------------------------------------------------------------------
template <int L, int PPT, bool SHORT>
__device__ __forceinline__ void tile_f64(const double *__restrict__ s_rec, int n, const double (&c)[PPT][3],
                                         double (&tacc)[PPT], const double *__restrict__ boys64)
{
    constexpr int st = rec64_stride(L);
    for (int j = 0; j < n; ++j) {
        const double *r = s_rec + j * st;
#pragma unroll
        for (int q = 0; q < PPT; ++q)
            tacc[q] += dist_f64<L, SHORT>(r, c[q][0], c[q][1], c[q][2], boys64);
    }
}

template <int NT, int PPT>
__device__ __forceinline__ void cta_f64(const EvalArgs &a, int bx, int split, float4 *smem4)
{
    const double *s_rec = reinterpret_cast<const double *>(smem4);
    const int base = bx * NT * PPT + threadIdx.x;
    double c[PPT][3], S[PPT], Cc[PPT];
    int idx[PPT];
#pragma unroll
    for (int q = 0; q < PPT; ++q) {
        int i = base + q * NT;
        idx[q] = i;
        int ic = min(i, a.n_pos - 1);
        c[q][0] = a.pos.x64[ic];
        c[q][1] = a.pos.y64[ic];
        c[q][2] = a.pos.z64[ic];
        S[q] = 0.0;
        Cc[q] = 0.0;
    }
    for (int t = split; t < a.n_tiles; t += a.n_splits) {
        const TileMeta m = a.tiles[t];
        __syncthreads();
        const bool pts = is_point_class(m.cls);
        const int nvec = pts ? m.n * 2 : (m.n * rec64_stride(m.cls & 7)) / 2;
        copy_tile(smem4, reinterpret_cast<const float4 *>(a.rec64 + m.off64), nvec);
        __syncthreads();
        double tacc[PPT];
#pragma unroll
        for (int q = 0; q < PPT; ++q)
            tacc[q] = 0.0;
        if (pts) {
            tile_points_f64<PPT>(s_rec, m.n, c, tacc);
        } else {
            switch (m.cls) {
            case 0: tile_f64<0, PPT, false>(s_rec, m.n, c, tacc, a.boys64); break;
            case 1: tile_f64<1, PPT, false>(s_rec, m.n, c, tacc, a.boys64); break;
            case 2: tile_f64<2, PPT, false>(s_rec, m.n, c, tacc, a.boys64); break;
            case 3: tile_f64<3, PPT, false>(s_rec, m.n, c, tacc, a.boys64); break;
            case 4: tile_f64<4, PPT, false>(s_rec, m.n, c, tacc, a.boys64); break;
            case 8: tile_f64<0, PPT, true>(s_rec, m.n, c, tacc, a.boys64); break;
            case 9: tile_f64<1, PPT, true>(s_rec, m.n, c, tacc, a.boys64); break;
            case 10: tile_f64<2, PPT, true>(s_rec, m.n, c, tacc, a.boys64); break;
            case 11: tile_f64<3, PPT, true>(s_rec, m.n, c, tacc, a.boys64); break;
            default: tile_f64<4, PPT, true>(s_rec, m.n, c, tacc, a.boys64); break;
            }
        }
#pragma unroll
        for (int q = 0; q < PPT; ++q)
            two_sum_acc(S[q], Cc[q], tacc[q]);
    }
#pragma unroll
    for (int q = 0; q < PPT; ++q)
        if (idx[q] < a.n_pos)
            a.partial[(size_t)split * a.n_pos + idx[q]] = S[q] + Cc[q];
}

template <int NT, int PPT>
__global__ void __launch_bounds__(NT) potential_f64_kernel(EvalArgs a)
{
    extern __shared__ float4 smem4[];
    cta_f64<NT, PPT>(a, blockIdx.x, blockIdx.y, smem4);
}

// ---------------------------------------------------------------------------
// Batched systems: persistent kernel over (system, position block, split)
// work items taken from an atomic counter, plus grid-stride staging and
// reduction over every system's positions.  All sizes and pointers come from
// the device-side table (BatchHeader + SysDesc[]), so one captured CUDA graph
// serves every call whose work fits the allocated capacity.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int find_sys(const SysDesc *__restrict__ sys, int n_sys, int pos)
{
    int lo = 0, hi = n_sys - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (sys[mid].pos_begin <= pos)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int find_group(const BatchGroup *__restrict__ groups, int n, int item)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (groups[mid].item_begin <= item)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ EvalArgs args_of(const SysDesc &d, const float *boys32, const double *boys64,
                                            const float *boysdd)
{
    EvalArgs a;
    a.n_pos = d.n_pos;
    a.n_splits = 1;
    a.tile_size = d.tile_size;
    a.pos = d.st;
    a.tiles = d.tiles;
    a.rec32 = d.rec32;
    a.rec64 = d.rec64;
    a.boys32 = boys32;
    a.boys64 = boys64;
    a.recdd = d.recdd;
    a.boysdd = boysdd;
    a.dd_lim = d.dd_lim;
    a.pairs = 0;
    a.near_r = d.near_r;
    return a;
}

template <int NT, int PPT, int PREC>
__global__ void __launch_bounds__(NT, PREC == 1 ? 512 / NT : 1) batch_potential_kernel(const BatchHeader *__restrict__ hdr,
                                                             const SysDesc *__restrict__ sys,
                                                             const BatchGroup *__restrict__ groups, int *counter,
                                                             const float *boys32, const double *boys64,
                                                             const float *boysdd, int tile_cap)
{
    extern __shared__ float4 smem4[];
    __shared__ int s_item;
    __shared__ double s_acc[PREC == 1 ? NT * PPT : 1];
    float *s_boys = reinterpret_cast<float *>(smem4 + (tile_cap * kRec32MaxStride) / 4);
    if (PREC == 1)
        for (int i = threadIdx.x; i < kBoys32Rows * kBoys32Row; i += NT)
            s_boys[i] = boys32[i];
    const int n_items = hdr->n_items, n_groups = hdr->n_groups;
    for (;;) {
        __syncthreads(); // s_item and the tile buffer are free again
        if (threadIdx.x == 0)
            s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= n_items)
            break;
        const BatchGroup g = groups[find_group(groups, n_groups, item)];
        const SysDesc &d = sys[g.sys];
        const int local = item - g.item_begin, range = local / d.blocks, bx = local % d.blocks;
        EvalArgs a = args_of(d, boys32, boys64, boysdd);
        const int t0 = int((long long)g.n_tiles * range / g.ranges), t1 = int((long long)g.n_tiles * (range + 1) / g.ranges);
        a.tiles = d.tiles + g.tile0 + t0;
        a.n_tiles = t1 - t0;
        a.partial = d.partial + (size_t)(g.split0 + range) * d.n_pos;
        single_group(a);
        if (PREC == 1)
            cta_f32c<NT, PPT, true>(a, bx, 0, smem4, s_boys, s_acc);
        else
            cta_f64<NT, PPT>(a, bx, 0, smem4);
    }
}

} // namespace

} // namespace esp
