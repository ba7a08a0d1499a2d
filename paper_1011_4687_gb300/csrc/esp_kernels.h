// Device-side launch interface of the potential kernels.
#pragma once

#include <cuda_runtime.h>

#include "esp_internal.h"

namespace esp {

// Recentred positions, structure of arrays: FP64 copy and FP32 hi + lo split,
// hi on the environment's coordinate grid and lo = fp32(x - hi), so FP32 code
// forms P - C as (P_hi - C_hi) + (P_lo - C_lo) with an exact first difference.
struct Staged {
    double *x64, *y64, *z64;
    float *xh, *yh, *zh, *xl, *yl, *zl;
    // the same rest x - hi in two words, mid on the grid 2^-23 q (esp_dd.h)
    float *xm, *ym, *zm, *xr, *yr, *zr;
};
constexpr size_t kStagedBytes = 3 * sizeof(double) + 12 * sizeof(float); // per position
// the arrays of n positions, one after the other from b (8-byte aligned)
inline Staged staged_at(void *b, size_t n)
{
    Staged st;
    st.x64 = static_cast<double *>(b);
    st.y64 = st.x64 + n;
    st.z64 = st.y64 + n;
    float *f = reinterpret_cast<float *>(st.z64 + n);
    float **p[] = {&st.xh, &st.yh, &st.zh, &st.xl, &st.yl, &st.zl, &st.xm, &st.ym, &st.zm, &st.xr, &st.yr, &st.zr};
    for (float **q : p) {
        *q = f;
        f += n;
    }
    return st;
}

// FP32C tile groups: FP64 point charges, FP32 point charges, then one group
// per L (long- and short-range tiles of that L together).
constexpr int kMaxTileGroups = 7;
constexpr int kMaxPartShift = 2; // tiles are dealt in up to four parts

struct EvalArgs {
    int n_pos;
    int n_splits;     // tiles are dealt round-robin to this many splits
    int n_tiles;
    int tile_size;
    Staged pos;
    const TileMeta *tiles;
    const float *rec32;
    const double *rec64;
    const float *boys32;
    const double *boys64;
    const float *recdd;   // dd records (TileMeta::offdd)
    const float *boysdd;  // Boys table of the dd general form
    float dd_lim;         // |coordinate| up to which the dd words of a position are exact
    double *partial;  // [n_splits][n_pos], 8 bytes each
    int pairs;        // FP32C kernel: its partials as float2 (sum, compensation), in the same places
    float near_r;     // FP32C: blocks closer than this to a tile's bounding sphere are left to the dd kernel
    // FP32C deal by tile group: group g holds tiles [grp_tile[g], grp_tile[g+1])
    // and takes the splits [grp_split[g], grp_split[g+1]) (grp_split[n_groups] =
    // n_splits), so each CTA runs the code of one class.  One group over all
    // tiles is the plain round-robin deal.
    int n_groups;
    int grp_tile[kMaxTileGroups + 1];
    int grp_split[kMaxTileGroups + 1];
    // A group's tiles are dealt in 2^grp_shift parts of tile_size >> grp_shift records.
    int grp_shift[kMaxTileGroups];
};

// the plain deal: every tile in one group over n_splits splits
ESP_HD void single_group(EvalArgs &a)
{
    a.n_groups = 1;
    a.grp_tile[0] = 0;
    a.grp_tile[1] = a.n_tiles;
    a.grp_split[0] = 0;
    a.grp_split[1] = a.n_splits;
    a.grp_shift[0] = 0;
}

// One system of a batched evaluation (device-side table entry).
struct SysDesc {
    const TileMeta *tiles;
    const float *rec32;
    const double *rec64;
    const float *recdd;   // null: FP64 code in place of the dd sums
    float dd_lim;
    const double *pos_in; // [n_pos][3] device
    double *V_out;        // [n_pos] device
    double *partial;      // [splits][n_pos]
    Staged st;
    double qm[3];
    double quantum;
    int n_tiles, tile_size, n_pos, splits, blocks, pos_begin;
    float near_r;
    int sorted;           // stage in spatial order (slot_of / perm below are [n_pos] scratch)
    int *slot_of, *perm;
};

// The work items of one tile group of one system: items item_begin + range *
// blocks + block, each range a contiguous part of the group's tiles with its own
// partial sums (split split0 + range).  Entries are ordered by class first, so
// that the CTAs of an SM run one class's code at a time.
struct BatchGroup {
    int item_begin, sys, tile0, n_tiles, ranges, split0;
};

struct BatchHeader {
    int n_sys, n_items, n_pos_total, n_groups;
};

// Batched pipeline on stream s: staging, persistent potential kernel over all
// (system, block, range of tiles) items, reduction into each system's V_out.  The
// counter must be zero when the potential kernel starts.
// max_sys: the number of systems (one spatial-order CTA each, for systems marked sorted)
cudaError_t launch_batch(int precision, const BatchHeader *hdr, const SysDesc *sys, const BatchGroup *groups,
                         int max_sys, int *counter,
                         int max_items,
                         const float *boys32, const double *boys64, const float *boysdd, int tile_cap, int threads,
                         int ppt,
                         int num_sms, int max_pos_total, cudaStream_t s);
bool batch_shape_supported(int precision, int threads, int ppt);

// The tiles list[0..n_list) (FP64 point charges, and the tiles that can be near
// a position, at their near positions) summed at FP64 accuracy into n_splits
// partial sums from a.partial on (esp_ddsum.cu).
int dd_sum_splits(int n, int n_list, int num_sms);
cudaError_t launch_dd_sum(const EvalArgs &a, const int *list, int n_list, int n_splits, cudaStream_t s);
// All tiles at FP64 accuracy into a.n_splits partial sums (esp_ddsum.cu): far
// entries in FP32 words, the others in FP64.
int td_splits(int n, int n_tiles, int num_sms, int &shift);
cudaError_t launch_td(const EvalArgs &a, cudaStream_t s);
// dd records (esp_dd.h) of the tiles with offdd >= 0, on the coordinate grid q
cudaError_t launch_dd_build(const TileMeta *tiles, int n_tiles, const double *rec64, double q, float *recdd,
                            cudaStream_t s);

// slot_of (optional, from launch_sort): the staged slot of each input position
cudaError_t launch_stage(const double *pos_in, int n, const double center[3], double quantum, const Staged &st,
                         cudaStream_t s, const int *slot_of = nullptr);
// Spatial order of n positions (stable counting sort by the Morton code of a
// 16^3 cell grid over [-8, 8]^3 bohr about center).  scratch holds
// sort_scratch_ints(n) ints; on return *slot_of[i] is the slot of position i
// and *perm[slot] its input index (both inside scratch).
constexpr int kSortSide = 16;
constexpr int kSortCells = kSortSide * kSortSide * kSortSide;
constexpr int kSortThreads = 1024;
constexpr int kSortCtas = 8; // the cluster that orders one call's positions
constexpr double kSortHalf = 8.0;
constexpr int kSortMinPositions = 4096; // fewer: the order is not worth its two launches
constexpr int kSortMinTd = 512;        // FP64: compact warps have fewer near entries
size_t sort_scratch_ints(int n);
cudaError_t launch_sort(const double *pos_in, int n, const double center[3], int *scratch, int **slot_of, int **perm,
                        cudaStream_t s);
// precision: 0 = FP64, 1 = FP32C.  threads in {64, 128, 256}, ppt in {1, 2, 4}.
cudaError_t launch_potential(int precision, const EvalArgs &a, int threads, int ppt, cudaStream_t s);
size_t potential_smem_bytes(int precision, int tile_size);
// A kernel's limit of dynamic shared memory belongs to the function, not to a
// launch: set to what kMaxTileSize takes, the same from every thread.  (Set to
// the calling context's own size, a thread with smaller tiles could lower it
// between another thread's set and launch, which then failed.)
constexpr int kMaxTileSize = 256;
template <typename K> inline cudaError_t allow_smem(K kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
// Launch shapes compiled into the library: FP64 threads {64,128,256} x ppt {1,2};
// FP32C (64,{2,4}), (128,{1,2,4}), (256,{1,2}).
bool potential_shape_supported(int precision, int threads, int ppt);
// Few positions per call (n <= kSmallN): environment entries spread over the
// threads of one launch, a chunk of up to kSmallChunk positions per CTA row.
// Entries are evaluated at FP64 accuracy (far ones in FP32 words), except the FP32 point charges (class
// kClassPoint32) when n_p32 is set: those take the compensated FP32 form of
// the main kernel (hi/lo offsets, symmetric rsqrt, low word of the charge),
// sum per thread in FP32 and across threads as (sum, compensation) pairs; the
// FP64 point charges beside them take the dd form.
constexpr int kSmallN = 128;
constexpr int kSmallChunk = 16;      // positions of one CTA
constexpr int kSmallThreads = 512;
constexpr int kSmallMaxChunks = (kSmallN + kSmallChunk - 1) / kSmallChunk;
constexpr int kSmallNDistributions = 16; // calls above this many positions take the
                                         // few-position path only for environments of point charges
struct SmallArgs {
    int n_pos;
    int n_tiles;
    const double *pos_in;  // [n_pos][3] device positions (recentred inside the kernel)
    double cx, cy, cz;     // QM centre
    const TileMeta *tiles;
    const double *rec64;
    const float *rec32;
    const float *recdd;
    const double *boys64;
    double quantum, inv_quantum; // coordinate grid of the FP32 hi words
    float dd_lim;
    int points_dd;         // FP64 point charges beside FP32 ones: as dd sums
    int any64;             // some entry is summed in FP64
    int64_t p32_off;       // float offset of the FP32 point records (contiguous, n_p32 of them)
    int n_p32;             // 0: every entry in FP64
    // the tiles outside the flat FP32 pass: n_other of them, tile o or, from
    // skip_begin on, o + n_skip, in tile_parts parts of 64 entries each
    int n_other, skip_begin, n_skip, tile_parts;
    int direct; // all of them in FP64, in parts of 32 entries
    int dist;   // some of them are distributions
    int *counters;         // [kSmallMaxChunks], zero before and after every launch
    // set by launch_small_n
    int g_threads;
    float2 *part32;
    double *part64;
};
// scratch of one launch
size_t small_n_bytes(int n_tiles, int num_sms, int n);
cudaError_t launch_small_n(SmallArgs a, void *scratch, int num_sms, double *V, cudaStream_t s);
// perm (optional, from launch_sort): V[perm[slot]] receives the sum of slot
// in_order: the partials one after the other (else several chains, joined);
// n64 >= 0: the partials after the first n64 as float2 (sum, compensation)
cudaError_t launch_reduce(const double *partial, int n_splits, int n, double *V, cudaStream_t s,
                          const int *perm = nullptr, bool in_order = false, int n64 = -1);
cudaError_t launch_walkers(const double *V, int n_walkers, int n_elec, double *E, cudaStream_t s);

} // namespace esp
