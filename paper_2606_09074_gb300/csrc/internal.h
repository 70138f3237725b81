// Host-side declarations of the kernel launchers.  Each launch_* enqueues
// exactly one kernel on `stream` and returns the launch error.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "refine.h"
#include "common.cuh"

namespace refine {

// Where a launcher puts its kernel: a stream, and whether the kernel may start
// its launch while the kernel before it in the stream ends (programmatic
// dependent launch; every kernel launched so waits for the earlier ones with
// pdl_wait before it touches memory).  The plain calls chain their kernels: a
// selection of 1.75M scores takes 29 instead of 43 us, a pass over 1M x 150
// 313 instead of 342 us.  The batch and the queue do not: kernels that wait on
// one stream would hold the SMs that another stream's could use.
struct Chain {
    cudaStream_t s;
    bool on = false;
    Chain(cudaStream_t stream) : s(stream) {}
    Chain(cudaStream_t stream, bool chained) : s(stream), on(chained) {}
};
template <typename... K, typename... A>
cudaError_t launch_chained(void (*k)(K...), int grid, int threads, size_t smem, const Chain &c, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c.s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = c.on ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, static_cast<K>(args)...);
}

// Cameras processed per score launch at most (80 bytes each in shared
// memory, 128 with REFINE_FLAG_FULL_JACOBIAN).  A larger view set is split into passes (camera blocks) of
// ScoreShape::views_per_pass views, a multiple of 32; a primitive's running
// Kahan pair (sum, compensation) is carried from pass to pass, so its sum
// is the same whatever the block size.
constexpr int kViewsPerPass = 512;
constexpr int kScoreThreads = 256;     // threads per CTA of k_score

// Work-item shape of the score kernels, chosen per device by the autotuner
// (refine_autotune).  Every primitive's score is computed by one thread with
// the views in a fixed order, whatever tile it is in, so the shape changes
// speed only, never a result.
struct ScoreShape {
    int gpt = 2;          // primitives per thread: a warp's tile is 32 * gpt primitives (1 or 2)
    int threads = 256;    // threads per CTA of the batched kernel (128 or 256); k_score uses kScoreThreads
    int ctas_per_sm = 0;  // cap on resident CTAs per SM of the batched kernel (0 = as many as fit)
    int views_per_pass = kViewsPerPass;  // camera block: views per score pass (32..512, a multiple of 32)
};
bool shape_valid(const ScoreShape &sh);
// Work of a scene in a batched launch, in (32-primitive, view) pairs.
inline long long batch_work(int64_t n, int vcount) { return (long long)((n + 31) / 32) * vcount; }
// CTAs of a batched launch over scenes of `tiles32` 32-primitive groups in
// all: no more than there are tiles for their warps.
inline int batch_grid(const ScoreShape &sh, int full_grid, long long tiles32)
{
    const long long per_cta = (long long)sh.gpt * (sh.threads / 32);
    const long long g = (tiles32 + per_cta - 1) / per_cta;
    return (int)(g < 1 ? 1 : (g < full_grid ? g : full_grid));
}

// Spatial cells for the processing order of k_score: a 2^b x 2^b x 2^b grid
// over the scene's mean +- 3 sigma box, numbered along a Hilbert curve, with b the
// largest value in [kMinCellBits, kMaxCellBits] that leaves ~0.5 primitives
// per cell or more (cell_bits_for).  Fine cells keep the counting sort's
// atomics spread out: dense scenes put hundreds of centres in one coarse
// cell, and atomics on one address serialise.
constexpr int kMinCellBits = 4;
constexpr int kMaxCellBits = 7;
constexpr int kScanThreads = 1024;
constexpr int kScanCells = 4 * kScanThreads;  // cells per block of the cell scan (4 per thread)
inline int cell_bits_for(int64_t n)
{
    int b = kMinCellBits;
    while (b < kMaxCellBits && (int64_t(1) << (3 * (b + 1))) <= n * 2) ++b;
    return b;
}
// Keys of the processing order: the cell, then, for the primitives with large
// scales (ln s_max > OrderGrid::big_ls), which thereby follow all the others,
// 2^(3b) plus a cell of a grid half as fine; rounded up to whole blocks of the
// cell scan.
inline int order_keys(int bits)
{
    const int keys = (1 << (3 * bits)) + (1 << (3 * (bits - 1)));
    return (keys + kScanCells - 1) / kScanCells * kScanCells;
}
constexpr float kSizeSplitSd = 1.28f;

// Diagnostic counters of k_score (written only when ScoreLaunch::need is set).
enum {
    kCntTiles = 0,     // (warp tile, view) classifications
    kCntInPairs,       // pairs in tiles classified entirely visible
    kCntOutPairs,      // pairs in tiles classified entirely invisible
    kCntMixedPairs,    // pairs evaluated one by one
    kCntBoundPairs,    // of those: centre outside the image, in the depth range
    kCntExactPairs,    // of those: within the conservative footprint radius
    kCntVisMixed,      // pairs evaluated one by one and found visible
    kCntOpenX,         // pairs evaluated one by one with the u axis open (U computed)
    kCntOpenY,         //   ... with the v axis open (V computed)
    kCntOpenZ,         //   ... with the depth range open (compared)
    kCntBoundX,        // bound-stage pairs with the u axis open
    kCntBoundY,        // bound-stage pairs with the v axis open
    kCntExactX,        // exact-stage pairs whose u extent was needed (centre beyond u)
    kCntExactY,        // exact-stage pairs whose v extent was needed
    kCntExactWarpAxes, // warp-level executions of one axis of the exact test
    kCountSlots
};

// Per-primitive record written by the feature pass, in scene order (64 B):
//   a = (mu.x, mu.y, mu.z, b2)   b2 = 9 s_max^2 (1 + 2^-10), the footprint
//                                bound factor; -(1 + b2) when a scale
//                                underflowed to 0
//   b, c, d.x = L, row-major 3x3 with rows 3 s_k r_k (r_k the k-th column of
//                R(q)), so that L^T L = 9 Sigma
//   d.y = alpha, d.z = m_gem, d.w = m_col
struct __align__(16) PrimRec {
    float4 a, b, c, d;
};
static_assert(sizeof(PrimRec) == 64, "primitive record layout");

// Projection mode of a set of flags (the weight of a visible pair).
enum { kProjEq17 = 0, kProjNone = 1, kProjFullJ = 2 };
__host__ __device__ inline int proj_mode(int flags)
{
    return (flags & REFINE_FLAG_NO_PROJ) ? kProjNone : (flags & REFINE_FLAG_FULL_JACOBIAN) ? kProjFullJ : kProjEq17;
}
// Shared memory of a camera block.
__host__ __device__ inline size_t cams_smem(int vcount, int flags)
{
    return (size_t)vcount * (sizeof(CamRec) + (proj_mode(flags) == kProjFullJ ? sizeof(CamExt) : 0));
}

struct ScoreLaunch {
    const PrimRec *recs;        // records in scene order
    int64_t n;
    const uint32_t *perm;       // processing order (a permutation of 0..n-1)
    const CamRec *cams;         // this pass's cameras (device, 16-byte aligned)
    const CamExt *ext;          // their extensions (FULL_JACOBIAN, else NULL)
    int vcount;                 // cameras in this pass
    int first, last;            // first / last pass of the view set
    float eta;
    float inv_views;            // 1 / |V|
    int flags;
    const SceneConsts *consts;
    float2 *running;            // per-primitive running (sum, Kahan compensation) between passes
    float *scores;
    float *view_sum;            // optional
    unsigned long long *need;   // optional diagnostic counters (kCountSlots), see k_score
    unsigned long long *tiles_taken;  // k_score: item counter, zero before the launch (required;
                                      // k_score_batch draws from BatchLaunch::next)
    int split_tiles;            // k_score: tiles taken in items of kSplitViews views (score_plan)
    float *parts;               //   their block sums, [split_tiles][blocks of the pass][tile]
    unsigned *parts_done;       //   items finished per split tile, zero before the launch
    int *status;
    int grid;                   // CTAs (persistent)
};

constexpr int kSplitViews = 64;  // views per item of a split tile, a multiple of 32
// How k_score runs a pass (score_plan): CTAs, primitives per thread, and the
// tiles at the end of the launch whose views are split into items.
struct ScorePlan {
    int grid = 1, gpt = 2, split_tiles = 0;
};
inline size_t split_part_floats(const ScorePlan &pl, int vcount)
{
    return (size_t)pl.split_tiles * ((vcount + 31) / 32) * 32 * pl.gpt;
}

// First kernel of a scene: the processing-order grid, the camera records of
// views 0, vstride, 2 vstride, ... (V of them), and two ranges to clear.
struct PrepLaunch {
    const refine_camera *cams;
    int V, vstride;
    CamRec *cam_out;
    CamExt *ext_out;  // NULL unless FULL_JACOBIAN
    int cell_bits;
    OrderGrid *grid;
    uint4 *zero, *more;  // 16-byte words to clear
    int64_t zero4, more4;
    int *status;
};
cudaError_t launch_prepare(const float *pos, const void *attr, int dtype, int64_t stride, int64_t n, const PrepLaunch &a,
                           int num_sms, const Chain &s);

struct FeatureLaunch {
    const float *pos;
    const void *attr;
    int64_t stride, n;
    float eta;
    const float *luma;  // host
    PrimRec *recs;
    float2 *partials;   // per block, float-float sums
    const OrderGrid *grid;
    int cell_bits;
    uint2 *cell;        // (key, slot) of every primitive
    unsigned *counts;   // per key, zero before the launch
    int *status;
};
int feature_blocks(int64_t n);
cudaError_t launch_features(const FeatureLaunch &f, int dtype, int num_sms, const Chain &s);

// What the cell scatter's first block forms from the feature pass's block sums.
struct SceneTail {
    const float2 *partials;
    int nblocks;
    int64_t n;
    refine_params p;
    SceneConsts *consts;
    SceneStats *stats;
};
cudaError_t launch_cell_scan(unsigned *counts, unsigned *off_local, unsigned *bsum, unsigned *done, int cell_bits,
                             const Chain &s);
cudaError_t launch_cell_scatter(const uint2 *cell, int64_t n,
                                const unsigned *off_local, const unsigned *bsum, uint32_t *perm,
                                const SceneTail &tail, int num_sms, const Chain &s);
cudaError_t launch_score(const ScoreLaunch &a, int gpt, const Chain &s);
// split: tiles may be split (the caller provides parts and parts_done).
ScorePlan score_plan(int num_sms, int64_t n, int vcount, int flags, bool split, const ScoreShape &sh);

// FP32 FMA throughput probe (refine_fma_rate): FLOPs of one launch of
// `iters` steps on `num_sms` SMs, and the launch itself (sink: one float,
// never written).
constexpr int kFmaProbeMaxIters = 1 << 20;  // about 65 ms at the nominal FP32 peak
double fma_probe_flops(int num_sms, int iters);
cudaError_t launch_fma_probe(int num_sms, int iters, float *sink, cudaStream_t s);

// Self-test of the bounded mbarrier wait (refine_selftest_wait).
constexpr uint32_t kSelftestMaxBytes = 1024;
cudaError_t launch_wait_selftest(const void *src, uint32_t bytes, uint32_t missing, long long limit, int *status,
                                 cudaStream_t s);

// Batched score launch over the tiles of many scenes (each scene a single
// pass of at most kViewsPerPass views).
struct BatchLaunch {
    const ScoreLaunch *scenes;       // device [n_scenes]
    const long long *work;           // device [n_scenes + 1], work of the scenes before each (batch_work)
    int n_scenes;
    unsigned *next;                  // device [n_scenes], tiles drawn of each, zero before the launch
    bool eq17;                       // every scene has the Eq. 17 projection mode
    int *status;
};
// smem: the largest camera block among the scenes (cams_smem).
int score_batch_grid(int num_sms, size_t smem, bool eq17, const ScoreShape &sh);
cudaError_t launch_score_batch(const BatchLaunch &b, size_t smem, int grid, const ScoreShape &sh, cudaStream_t s);

// ------------------------------------------------------------- select
struct SelState {
    unsigned int hist[2048];
    unsigned int done;
    unsigned int prefix;
    unsigned int remaining;
    unsigned int kstar;
    unsigned int need_ties;
    unsigned int pad[3];
    long long idx_cut;
};
// Up to this many scores the selection is one cluster launch
// (launch_select_cluster, which needs nothing cleared and only kstar of the
// state); above it, the passes below, also where they are chained (then they
// take 22.5-23 us instead of 34 up to 400k scores).
constexpr int64_t kSelClusterMax = 8 * 32 * 1024;
constexpr int64_t kSelClusterChained = 128 * 1024;
cudaError_t launch_select_cluster(const float *scores, int64_t n, uint32_t n_keep, SelState *st, uint32_t *mask,
                                  int *status, const Chain &s);
constexpr int kTieSeg = 4096;
int select_grid(int num_sms, int64_t n);
cudaError_t launch_select_pass(int pass, const float *scores, int64_t n, uint32_t n_keep,
                               SelState *st, bool vec, int grid, int *status, const Chain &s);
cudaError_t launch_select_ties(const float *scores, int64_t n, SelState *st, unsigned *seg_cnt,
                               int grid, const Chain &s);
cudaError_t launch_select_mask(const float *scores, int64_t n, const SelState *st, uint32_t *mask,
                               int num_sms, const Chain &s);
cudaError_t launch_mask_fill(uint32_t *mask, int64_t n, const Chain &s);

// ------------------------------------------------------------- compact
struct CmpState {
    unsigned int done;
    unsigned int ok;
    long long total;
};
constexpr int kCmpSeg = 256;        // elements per compaction segment (8 mask words)
constexpr int kCmpBlockSegs = 256;  // segments per block of launch_compact_local (65,536 elements)
constexpr int kCmpMaxBlocks = 256;  // its blocks at most (16.8M elements)
inline int cmp_blocks(int64_t n) { return (int)((n + (int64_t)kCmpSeg * kCmpBlockSegs - 1) / (kCmpSeg * kCmpBlockSegs)); }
// Where the segments' kept elements go: offsets within blocks and the blocks'
// totals (blocks > 0), or offsets in the whole output.
struct CmpOffsets {
    int blocks;
    const unsigned *local, *totals;
    const unsigned long long *global;
    CmpState *state;
};
cudaError_t launch_compact_local(const uint32_t *mask, int64_t n, unsigned *local, unsigned *totals, const Chain &s);
cudaError_t launch_compact_count(const uint32_t *mask, int64_t n, unsigned *seg_cnt,
                                 unsigned long long *seg_off, CmpState *cs, int64_t out_stride,
                                 int grid, int *status, const Chain &s);
cudaError_t launch_compact_scatter(const refine_scene &in, const uint32_t *mask, const CmpOffsets &off, float *out_pos,
                                   void *out_attr, int64_t out_stride, int32_t *out_idx, int num_sms, int *status,
                                   const Chain &s);

}  // namespace refine
