// Preparation kernels: camera records, the content-feature pass (Eq.
// (features), Eq. 18-19) with the primitive records, and the spatial
// processing order of the score kernels.
#include <float.h>
#include <math.h>

#include "internal.h"
#include "rows.cuh"

namespace refine {

// ---------------------------------------------------------------------
// Camera preparation: refine_camera -> CamRec (P = K W and p = K t formed
// in double and rounded once), with validation.
// ---------------------------------------------------------------------
__device__ void prep_camera(const refine_camera *__restrict__ cams, int v, int vstride, CamRec *__restrict__ out,
                            CamExt *__restrict__ ext, int *status)
{
    refine_camera c = cams[(int64_t)v * vstride];
    bool ok = isfinite(c.fx) && isfinite(c.fy) && isfinite(c.cx) && isfinite(c.cy) &&
              isfinite(c.znear) && isfinite(c.zfar) && c.fx > 0.f && c.fy > 0.f &&
              c.width >= 1 && c.height >= 1 && c.znear > 0.f && c.zfar > c.znear;
    for (int k = 0; k < 9; ++k) ok = ok && isfinite(c.R[k]);
    for (int k = 0; k < 3; ++k) ok = ok && isfinite(c.t[k]);
    CamRec r;
    if (!ok) {
        set_status(status, kEinval);
        r.r0 = make_float4(0.f, 0.f, 0.f, 0.f);
        r.r1 = r.r2 = r.k = r.r0;
        r.lim = make_float4(0.f, 0.f, 1.f, 0.f);  // znear > zfar: never visible
        out[v] = r;
        if (ext) ext[v] = CamExt{r.r0, r.r0, r.r0};
        return;
    }
    double fx = c.fx, fy = c.fy, cx = c.cx, cy = c.cy;
    r.r0 = make_float4((float)(fx * c.R[0] + cx * c.R[6]), (float)(fx * c.R[1] + cx * c.R[7]),
                       (float)(fx * c.R[2] + cx * c.R[8]), (float)(fx * c.t[0] + cx * c.t[2]));
    r.r1 = make_float4((float)(fy * c.R[3] + cy * c.R[6]), (float)(fy * c.R[4] + cy * c.R[7]),
                       (float)(fy * c.R[5] + cy * c.R[8]), (float)(fy * c.t[1] + cy * c.t[2]));
    r.r2 = make_float4(c.R[6], c.R[7], c.R[8], c.t[2]);
    const float w = (float)c.width, h = (float)c.height;
    r.lim = make_float4(w, h, c.znear, c.zfar);
    // The edge norms Ex, Ey of the footprint bound (classify), rounded up;
    // the bound needs orthonormal rows of R (to well within the 2^-11 that the
    // primitives' s3 carries), so other cameras get none (every open pair
    // runs the exact test).
    float dot[6];
    for (int i = 0, k = 0; i < 3; ++i)
        for (int j = i; j < 3; ++j, ++k) {
            const float *a = c.R + 3 * i, *b = c.R + 3 * j;
            dot[k] = fmaf(a[0], b[0], fmaf(a[1], b[1], a[2] * b[2])) - (i == j ? 1.f : 0.f);
        }
    bool ortho = true;
    for (int k = 0; k < 6; ++k) ortho = ortho && fabsf(dot[k]) <= 1.220703125e-4f;  // 2^-13
    const float ex = fmaxf(fabsf(c.cx), fabsf(w - c.cx)), ey = fmaxf(fabsf(c.cy), fabsf(h - c.cy));
    const float Ex = sqrtf(fmaf(c.fx, c.fx, ex * ex)) * 1.00001f, Ey = sqrtf(fmaf(c.fy, c.fy, ey * ey)) * 1.00001f;
    // tile slack of the forms U, V, U - w z, V - h z (classify)
    float ca = 0.f, c0 = 0.f;
    for (const float4 &q : {r.r0, r.r1}) {
        ca = fmaxf(ca, fmaxf(fabsf(q.x), fmaxf(fabsf(q.y), fabsf(q.z))));
        c0 = fmaxf(c0, fabsf(q.w));
    }
    const float wh = fmaxf(w, h);
    ca = fmaxf(ca, wh * fmaxf(fabsf(r.r2.x), fmaxf(fabsf(r.r2.y), fabsf(r.r2.z))));
    c0 = fmaxf(c0, wh * fabsf(r.r2.w));
    r.k = make_float4(ortho ? Ex : FLT_MAX, ortho ? Ey : FLT_MAX, 2.f * kTileSlack * ca, 2.f * kTileSlack * c0);
    out[v] = r;
    if (ext) {
        CamExt e;
        e.tx = make_float4((float)(fx * c.R[0]), (float)(fx * c.R[1]), (float)(fx * c.R[2]), (float)(fx * c.t[0]));
        e.ty = make_float4((float)(fy * c.R[3]), (float)(fy * c.R[4]), (float)(fy * c.R[5]), (float)(fy * c.t[1]));
        e.f = make_float4((float)(fx * fx), (float)(fy * fy), 0.f, 0.f);
        ext[v] = e;
    }
}

// ---------------------------------------------------------------------
// Processing order.  Primitives are sorted by their cell in a 2^b x 2^b x
// 2^b grid over the mean +- 3 sigma box of the centres, cells numbered along
// a Hilbert curve (a counting sort: count, scan, scatter), so that the 32
// lanes of a warp hold nearby primitives and tend to take the same side of
// each view's frustum edges.  The primitives with the largest scales (ln
// s_max above mean + 1.28 sd, about the largest 10 % for a normal spread)
// come after all the others, in cells of their own, twice as wide, so that a
// tile's footprint bound (set by its largest s_max) is not set by a few large
// primitives among small ones.  The order only affects speed: every
// primitive's score is computed by one thread with the views in a fixed
// order, whatever its position, so the sort need not be stable (the
// count atomics order the primitives of a cell arbitrarily), and the grid box
// may come from a sample.
//
// Hilbert, not Morton order: neighbours along the curve are neighbours in
// space, so the boxes of 64 consecutive primitives are smaller.  MIXED pairs
// fall from 22.3 to 19.3 % (3.5M x 250 core-shell), 32.9 to 28.9 % (1M x
// 150) and 51.3 to 44.2 % (150k x 1100).  Finer grids (2^8, 2^10 per axis) and
// equal-mass cells gave no better tiles in a simulation.
// ---------------------------------------------------------------------
// Hilbert curve as a state machine (Hamilton's formulation: a state is the
// entry corner e and the axis d of a cube; octant o of the cube is its w-th
// along the curve): two levels per step.
struct HilbertTable {
    uint16_t t[24 * 64];  // [state][octant of level 1 << 3 | octant of level 2] -> next state << 6 | w1 << 3 | w2
};

constexpr HilbertTable make_hilbert_table()
{
    HilbertTable r{};
    int w1[24][8] = {}, nx[24][8] = {};
    for (int e = 0; e < 8; ++e)
        for (int d = 0; d < 3; ++d)
            for (int o = 0; o < 8; ++o) {
                const int k = (d + 1) % 3, x = o ^ e;
                const int l = ((x >> k) | (x << (3 - k))) & 7;  // rotate right by d + 1
                const int w = l ^ (l >> 1) ^ (l >> 2);          // inverse Gray code
                const int p = w == 0 ? 0 : 2 * ((w - 1) / 2);
                const int g = p ^ (p >> 1);  // entry corner of the w-th octant
                int dir = 0;
                if (w > 0)
                    for (int i = w % 2 == 0 ? w - 1 : w; i & 1; i >>= 1) ++dir;
                w1[e * 3 + d][o] = w;
                nx[e * 3 + d][o] = (e ^ (((g << k) | (g >> (3 - k))) & 7)) * 3 + (d + dir % 3 + 1) % 3;
            }
    for (int s = 0; s < 24; ++s)
        for (int a = 0; a < 8; ++a)
            for (int b = 0; b < 8; ++b)
                r.t[s * 64 + a * 8 + b] = (uint16_t)(nx[nx[s][a]][b] << 6 | w1[s][a] << 3 | w1[nx[s][a]][b]);
    return r;
}

__device__ const HilbertTable kHilbert = make_hilbert_table();

__device__ __forceinline__ void load_hilbert(uint16_t *smem)
{
    for (int k = threadIdx.x; k < 24 * 32; k += blockDim.x)
        reinterpret_cast<uint32_t *>(smem)[k] = __ldg(reinterpret_cast<const uint32_t *>(kHilbert.t) + k);
}

// Index of the cell (x, y, z), each below 2^8, along the curve.  Leading zero
// levels contribute zero digits, so it is below 2^(3b) for coordinates below
// 2^b (the orientation of the curve then depends on b, which does not matter).
__device__ __forceinline__ uint32_t hilbert_index(const uint16_t *t, uint32_t x, uint32_t y, uint32_t z)
{
    uint32_t h = 0, state = 0;
#pragma unroll
    for (int k = 6; k >= 0; k -= 2) {
        const uint32_t a = (x >> k) & 3u, b = (y >> k) & 3u, c = (z >> k) & 3u;  // two levels
        const uint32_t o = ((a >> 1) | (b & 2u) | ((c & 2u) << 1)) << 3 | (a & 1u) | ((b & 1u) << 1) | ((c & 1u) << 2);
        const uint32_t e = t[state * 64 + o];
        h = h << 6 | (e & 63u);
        state = e >> 6;
    }
    return h;
}

__device__ __forceinline__ uint32_t quantise(float x, float lo, float qs, float top)
{
    return (uint32_t)fminf(fmaxf((x - lo) * qs, 0.f), top);
}

// Key of a primitive: its cell, the large primitives (ls > big_ls) in cells
// twice as wide after all the others.
__device__ __forceinline__ uint32_t order_key(const uint16_t *hilbert, const OrderGrid &c, int cell_bits, float x, float y,
                                              float z, float ls)
{
    const float top = (float)((1 << cell_bits) - 1);
    const int big = ls > c.big_ls ? 1 : 0;
    const uint32_t h = hilbert_index(hilbert, quantise(x, c.lo[0], c.qscale[0], top) >> big,
                                     quantise(y, c.lo[1], c.qscale[1], top) >> big,
                                     quantise(z, c.lo[2], c.qscale[2], top) >> big);
    return h + (big ? 1u << (3 * cell_bits) : 0u);
}

// ---------------------------------------------------------------------
// First kernel of a scene.  Block 0 forms the processing-order grid from a
// sample of up to 1,024 primitives, 256 evenly spaced groups of four (one SM
// reads the six rows' sectors in a microsecond or two; 4,096 single ones took
// it over ten); the other blocks form the camera records and clear the cell counts
// and the score kernel's counters, which takes the place of two memsets.
// With the grid known beforehand, the feature pass counts the cells itself:
// the separate pass over positions and log-scales that did it took 60 us of
// a 3.5M-primitive scene, most of it waiting for its count atomics.
// ---------------------------------------------------------------------
constexpr int kPrepThreads = 1024;
constexpr float kGridFar = 6.f;  // standard deviations
constexpr int kGridRounds = 5;

template <int DT>
__global__ void __launch_bounds__(kPrepThreads) k_prepare(const float *__restrict__ pos, AttrRows<DT> attr, int64_t S,
                                                          int64_t n, PrepLaunch a)
{
    pdl_wait();  // never chained itself; lets the next kernel's launch begin
    if (blockIdx.x > 0) {
        const int64_t b = blockIdx.x - 1, nb = gridDim.x - 1;
        for (int64_t v = b + nb * threadIdx.x; v < a.V; v += nb * kPrepThreads)
            prep_camera(a.cams, (int)v, a.vstride, a.cam_out, a.ext_out, a.status);
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        for (int64_t i = b * kPrepThreads + threadIdx.x; i < a.zero4; i += nb * kPrepThreads) a.zero[i] = zero;
        for (int64_t i = b * kPrepThreads + threadIdx.x; i < a.more4; i += nb * kPrepThreads) a.more[i] = zero;
        return;
    }
    // Sums of the offsets from primitive 0 and of their squares (a scene far
    // from the origin keeps its digits), and of ln s_max.  A sample beyond
    // kGridFar standard deviations (at most 1 in 36 can be, none in an ordinary
    // scene) is left out and the sums are formed again about the mean found, as
    // long as that halves some deviation (a round is 1 us):
    // one centre of 1M at 1,000 or 10,000 scene radii among the 1,024 made the
    // box, and with it all cells, so much wider that a pass over 60 views took
    // 306 or 761 us, against 155 without it and 157 so.
    const int64_t k = threadIdx.x < n ? threadIdx.x : 0;
    const int64_t i = n <= kPrepThreads ? k : (k / 4) * (n - 4) / (kPrepThreads / 4 - 1) + k % 4;
    float base[4] = {__ldg(pos), __ldg(pos + S), __ldg(pos + 2 * S), 0.f};
    const float p[4] = {__ldg(pos + i), __ldg(pos + S + i), __ldg(pos + 2 * S + i),
                        fmaxf(attr.ld(0, i), fmaxf(attr.ld(1, i), attr.ld(2, i)))};
    bool use = threadIdx.x < n;
    int m = n < kPrepThreads ? (int)n : kPrepThreads;
    __shared__ float red[8][kPrepThreads / 32];
    __shared__ float sum[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float before[4] = {0.f, 0.f, 0.f, 0.f}, im;  // the variances found last, 1 / m
    for (int round = 0;; ++round) {
        float s[8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float v = use ? p[q] - base[q] : 0.f;
            s[q] = v;
            s[4 + q] = v * v;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
            if (lane == 0) red[q][warp] = s[q];
        }
        __syncthreads();
        if (warp < 8) {
            float t = red[warp][lane];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) sum[warp] = t;
        }
        __syncthreads();
        // (a reciprocal that is a little off moves the line by as little; by
        // division it took all threads a microsecond)
        im = rcp_approx_ftz((float)m);
        float mean[4];
        bool far = false, shrunk = round == 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            mean[q] = sum[q] * im;
            const float var = fmaf(-mean[q], mean[q], sum[4 + q] * im), d = (p[q] - base[q]) - mean[q];
            far |= use & (var > 0.f) & (d * d > kGridFar * kGridFar * var);
            shrunk |= 4.f * var < before[q];
            before[q] = var;
        }
        if (!shrunk || round == kGridRounds) break;  // (the same in every thread)
        const int dropped = __syncthreads_count(far);  // (every thread has read the sums)
        if (round == 0 && dropped == 0) break;
        use &= !far;
        m -= dropped;
#pragma unroll
        for (int q = 0; q < 4; ++q) base[q] += mean[q];
    }
    if (warp == 1 && lane < 4) {  // (beside the warps that look for crowds)
        const int q = lane;  // x, y, z, ln s_max
        const float mean = sum[q] / (float)m, var = sum[4 + q] / (float)m - mean * mean;
        const float sd = var > 0.f ? sqrtf(var) : 0.f;
        const float b = q == 0 ? base[0] : (q == 1 ? base[1] : (q == 2 ? base[2] : base[3]));
        if (q < 3) {
            a.grid->lo[q] = b + (mean - 3.f * sd);
            a.grid->qscale[q] = sd > 0.f && isfinite(sd) ? (float)(1 << a.cell_bits) / (6.f * sd) : 0.f;
        } else {
            const float big = b + (mean + kSizeSplitSd * sd);
            a.grid->big_ls = isfinite(big) ? big : INFINITY;
        }
    }
    // Whether cells are crowded: in two of four warps three samples or more
    // share one (by chance, every fifth of a scene whose fullest cell holds 5 %;
    // cells of an ordinary scene hold less than 0.01 %).  All 32 warps would take
    // 2 us: a match takes a step for each distinct value.
    bool crowd = false;
    if (warp % 8 == 0) {
        uint32_t cell = 0u;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float cells = (float)(1 << a.cell_bits), var = before[q];
            const float at = ((p[q] - base[q]) - sum[q] * im) * (var > 0.f ? rsqrtf(var) : 0.f);  // in sd
            cell = cell << 8 | (uint32_t)fminf(fmaxf((at + 3.f) * cells / 6.f, 0.f), cells - 1.f);
        }
        const unsigned peers = __match_any_sync(0xffffffffu, threadIdx.x < n ? cell : 0xffffff00u + lane);
        crowd = __any_sync(0xffffffffu, __popc(peers) >= 3);
    }
    const int crowds = __syncthreads_count(crowd);
    if (threadIdx.x == 0) a.grid->crowded = crowds >= 2 * 32;
}

cudaError_t launch_prepare(const float *pos, const void *attr, int dtype, int64_t stride, int64_t n, const PrepLaunch &a,
                           int num_sms, const Chain &s)
{
    // 4 stores of 16 bytes a thread, at most 64 cameras a block
    int64_t g = (a.zero4 + a.more4 + 4 * kPrepThreads - 1) / (4 * kPrepThreads);
    if (g < (a.V + 63) / 64) g = (a.V + 63) / 64;
    if (g > 2 * num_sms) g = 2 * num_sms;
    if (g < 1) g = 1;
    const int grid = (int)g + 1;
    if (dtype == REFINE_BF16)
        return launch_chained(k_prepare<REFINE_BF16>, grid, kPrepThreads, 0, s, pos, AttrRows<REFINE_BF16>(attr, stride),
                              stride, n, a);
    if (dtype == REFINE_BF16S)
        return launch_chained(k_prepare<REFINE_BF16S>, grid, kPrepThreads, 0, s, pos,
                              AttrRows<REFINE_BF16S>(attr, stride), stride, n, a);
    return launch_chained(k_prepare<REFINE_F32>, grid, kPrepThreads, 0, s, pos, AttrRows<REFINE_F32>(attr, stride), stride,
                          n, a);
}

// ---------------------------------------------------------------------
// Content features, primitive records and cell counts: one primitive per
// thread, its 59 rows read with coalesced loads (all in flight at once), its
// record and its feature terms formed (primitive_record), its cell counted.
// What bounds it is bytes: 236 / 124 / 130 read and 72 written a primitive.
// The count's slot comes back while the next primitive's rows are read.
// Counting here instead of in a pass of its own that read positions and
// log-scales again and waited for its atomics: 180 us against 188 + 60 us
// (3.5M float32), 156 against 160 + 58 us (bfloat16), 66 against 78 + 31 us
// (1M float32).  Streaming the SH rows with 16-byte loads of four primitives a
// lane, through shared memory and block barriers, took 244, 173 and 83 us.
//
// The sums of a scene are those of 256 x G threads (G = feature_blocks(n))
// that each take every (256 G)-th primitive in turn, in float, then a fixed
// float-float tree: their bits depend on n only.
// ---------------------------------------------------------------------
constexpr int kFeatCol = 256;                         // threads that take part in a block's sums
constexpr int kFeatCols = 8;                          // primitives per such thread at least, in a full grid
constexpr int kFeatRedLanes = 16;                     // threads per sum in the block reduction
constexpr int kFeatRedRow = kFeatCol + kFeatRedLanes; // padded row: two sums of a warp hit
                                                      // different banks
static_assert(kFeatSums * kFeatRedLanes <= kFeatCol, "one reduction thread per (sum, lane)");

template <int DT>
struct FeatureArgs {
    const float *pos;
    AttrRows<DT> attr;
    int64_t S, n;
    float eta, l0, l1, l2;
    PrimRec *recs;
    float2 *partials;
    const OrderGrid *grid;
    int cell_bits;
    uint2 *cell;
    unsigned *counts;
    int *status;

};

// Block sums in float-float: thread (k, j) adds the values of threads
// j, j + 16, j + 32, ... of sum k in that order, then the 16 lanes of
// sum k meet in a shuffle tree (xor 8, 4, 2, 1).
__device__ __forceinline__ void feature_block_sums(const float *red, float2 *partials)
{
    if (threadIdx.x < kFeatSums * kFeatRedLanes) {
        const int k = threadIdx.x / kFeatRedLanes, j = threadIdx.x % kFeatRedLanes;
        const float *col = red + k * kFeatRedRow + j;
        FF v = {col[0], 0.f};
#pragma unroll
        for (int q = kFeatRedLanes; q < kFeatCol; q += kFeatRedLanes) v = ff_add(v, FF{col[q], 0.f});
        // lanes of other sums in the same warp run the same tree on their own
        // 16-lane groups (xor below 16 stays within a group); the last warp
        // may hold reduction threads in its low lanes only
        constexpr int kRedThreads = kFeatSums * kFeatRedLanes;
        const unsigned lanes = (int)(threadIdx.x | 31u) < kRedThreads ? 0xffffffffu : (1u << (kRedThreads & 31)) - 1u;
#pragma unroll
        for (int o = kFeatRedLanes / 2; o > 0; o >>= 1)
            v = ff_add(v, FF{__shfl_xor_sync(lanes, v.hi, o), __shfl_xor_sync(lanes, v.lo, o)});
        if (j == 0) partials[(int64_t)blockIdx.x * kFeatSums + k] = make_float2(v.hi, v.lo);
    }
}

// What one primitive adds to the sums.
struct FeatTerms {
    float y, gem, mg, mc, alpha;
};

// The rows of one primitive: |SH|^2 summed row by row, and the others.
struct PrimRows {
    float sq, x, y, z, ls0, ls1, ls2, q0, q1, q2, q3, logit, dc0, dc1, dc2;
};

template <typename L>
__device__ __forceinline__ PrimRows read_rows(L &&ld)  // ld(r): row r of 59
{
    PrimRows p;
    p.sq = 0.f;
#pragma unroll
    for (int r = 11; r < 59; ++r) {
        const float x = ld(r);
        if (r == 11) p.dc0 = x;
        if (r == 12) p.dc1 = x;
        if (r == 13) p.dc2 = x;
        p.sq = fmaf(x, x, p.sq);
    }
    p.x = ld(0); p.y = ld(1); p.z = ld(2);
    p.ls0 = ld(3); p.ls1 = ld(4); p.ls2 = ld(5);
    p.q0 = ld(6); p.q1 = ld(7); p.q2 = ld(8); p.q3 = ld(9);
    p.logit = ld(10);
    return p;
}

// The next slot of a primitive's cell.  Where the cells are crowded (k_prepare)
// the lanes of a warp that share one take their slots in one add: adds to one
// address are served one by one.  Elsewhere there is nothing to share, and the
// search for it would take 1 us of 400k primitives.
__device__ __forceinline__ unsigned take_slot(unsigned *counts, unsigned key, int crowded)
{
    if (!crowded) return atomicAdd(&counts[key], 1u);
    const unsigned peers = __match_any_sync(__activemask(), key);
    const int lead = __ffs(peers) - 1, lane = threadIdx.x & 31;
    unsigned first = 0u;
    if (lane == lead) first = atomicAdd(&counts[key], (unsigned)__popc(peers));
    return __shfl_sync(peers, first, lead) + __popc(peers & ((1u << lane) - 1u));
}

template <int DT>
__device__ __forceinline__ FeatTerms feature_one(const FeatureArgs<DT> &f, const uint16_t *hilbert, const OrderGrid &og,
                                                 int64_t i, const PrimRows &p, float &bad, bool &zero_q, uint2 &key_slot)
{
    float4 ra, rb, rc, rd;
    FeatTerms t;
    bad = primitive_record(bad, p.x, p.y, p.z, p.ls0, p.ls1, p.ls2, p.q0, p.q1, p.q2, p.q3, p.logit, p.sq, f.eta, ra, rb,
                           rc, rd, t.gem, zero_q);
    t.y = luma_term(f.l0, f.l1, f.l2, p.dc0, p.dc1, p.dc2);
    t.alpha = rd.y;
    t.mg = rd.z;
    t.mc = rd.w;
    PrimRec *r = f.recs + i;
    r->a = ra; r->b = rb; r->c = rc; r->d = rd;
    key_slot.x = order_key(hilbert, og, f.cell_bits, p.x, p.y, p.z, fmaxf(p.ls0, fmaxf(p.ls1, p.ls2)));
    key_slot.y = take_slot(f.counts, key_slot.x, og.crowded);
    return t;
}

// Primitive i's rows by loads of its own (coalesced over the warp).
template <int DT>
__device__ __forceinline__ PrimRows load_rows(const FeatureArgs<DT> &f, int64_t i)
{
    return read_rows([&](int r) { return r < 3 ? __ldg(f.pos + r * f.S + i) : f.attr.ld(r - 3, i); });
}

// The sums of one thread.
struct FeatAcc {
    float s[kFeatSums];
    __device__ __forceinline__ void add(const FeatTerms &t)
    {
        s[0] += t.y;
        s[1] = fmaf(t.y, t.y, s[1]);
        s[2] = fmaf(t.alpha, 1.f - t.alpha, s[2]);
        s[3] += t.gem;
        s[4] += t.mg;
        s[5] += t.mc;
        s[6] += t.alpha;
    }
};

template <int DT>
__global__ void __launch_bounds__(kFeatCol, 4) k_features(FeatureArgs<DT> f)
{
    after(pdl_wait(), f.grid);  // the rows are older than the kernel before this one
    __shared__ float red[kFeatSums * kFeatRedRow];
    __shared__ __align__(4) uint16_t hilbert[24 * 64];
    load_hilbert(hilbert);
    const OrderGrid og = *f.grid;
    __syncthreads();
    FeatAcc acc = {};
    float bad = 0.f;
    bool zero_q = false;
    uint2 ks = make_uint2(0u, 0u);
    int64_t last = -1;  // its (key, slot) is stored in the next turn
    for (int64_t i = (int64_t)blockIdx.x * kFeatCol + threadIdx.x; i < f.n; i += (int64_t)gridDim.x * kFeatCol) {
        uint2 next;
        const FeatTerms t = feature_one<DT>(f, hilbert, og, i, load_rows<DT>(f, i), bad, zero_q, next);
        if (last >= 0) f.cell[last] = ks;
        ks = next;
        last = i;
        acc.add(t);
    }
    if (last >= 0) f.cell[last] = ks;
    if (!isfinite(bad)) set_status(f.status, kEnonfinite);
    if (zero_q) set_status(f.status, kEinval);
#pragma unroll
    for (int k = 0; k < kFeatSums; ++k) red[k * kFeatRedRow + threadIdx.x] = acc.s[k];
    __syncthreads();
    feature_block_sums(red, f.partials);
}

// The same with the rows of 256 primitives at a time brought into shared
// memory by bulk copies (RowTile), for bfloat16 rows: their 2-byte loads, 64
// bytes a warp, leave too few bytes in flight (four CTAs' tiles are 130 KB an
// SM).  The next tile is issued as soon as every thread has read the current
// one, so it arrives while the records are formed.  ALIGNED: every row starts
// on 16 bytes (the stride is a multiple of 8), so places are constants.  3.5M
// bfloat16 primitives: 157 -> 139 us (4.9 TB/s; what is left is the latency of
// a primitive's arithmetic at 32 warps an SM); the same with all copies issued
// by one warp 160 us.
template <int DT, bool ALIGNED>
__global__ void __launch_bounds__(kFeatCol, 4) k_features_bulk(FeatureArgs<DT> f, RowTile<DT, kFeatCol> in)
{
    using Rows = RowTile<DT, kFeatCol>;
    extern __shared__ __align__(16) unsigned char tile[];
    __shared__ float red[kFeatSums * kFeatRedRow];
    __shared__ __align__(4) uint16_t hilbert[24 * 64];
    __shared__ __align__(8) uint64_t bar;
    __shared__ int row_base[59];
    load_hilbert(hilbert);
    const int t = threadIdx.x;
    if (!ALIGNED && t < 59) row_base[t] = Rows::place(t) + (int)in.mis(t);
    if (t == 0) mbar_init(&bar, 1);
    after(pdl_wait(), f.grid);  // the rows are older than the kernel before this one
    const OrderGrid og = *f.grid;
    __syncthreads();
    auto stage = [&](int64_t i0) {
        const int count = (int)min((int64_t)kFeatCol, f.n - i0);
        in.template stage<kFeatCol / 32>(tile, i0, count, &bar);
        if (!ALIGNED && Rows::at_end(i0, f.n)) in.template rest<kFeatCol / 32>(tile, i0, count);
    };
    FeatAcc acc = {};
    float bad = 0.f;
    bool zero_q = false;
    uint2 ks = make_uint2(0u, 0u);
    int64_t last = -1;  // its (key, slot) is stored in the next turn
    const int64_t step = (int64_t)gridDim.x * kFeatCol;
    uint32_t phase = 0;
    int64_t i0 = (int64_t)blockIdx.x * kFeatCol;
    if (i0 < f.n) stage(i0);
    for (; i0 < f.n; i0 += step) {
        if (!ALIGNED && Rows::at_end(i0, f.n)) __syncthreads();  // what plain loads brought
        if (!mbar_wait_bounded(&bar, phase)) {
            set_status(f.status, kEtimeout);
            mbar_wait_bounded(&bar, phase);  // give the copies a second bound before leaving
            // the kernels that follow index with the slots: any valid ones
            if (last >= 0) f.cell[last] = ks;
            for (int64_t i = i0 + t; i < f.n; i += step) f.cell[i] = make_uint2(0u, atomicAdd(&f.counts[0], 1u));
            return;
        }
        phase ^= 1u;
        const PrimRows p = read_rows([&](int r) {
            const unsigned char *a = tile + (ALIGNED ? Rows::place(r) : row_base[r]) + Rows::size(r) * t;
            return Rows::f32(r) ? *reinterpret_cast<const float *>(a)
                                : __uint_as_float((uint32_t)*reinterpret_cast<const unsigned short *>(a) << 16);
        });
        __syncthreads();  // the tile is free
        if (i0 + step < f.n) stage(i0 + step);
        const int64_t i = i0 + t;
        if (i < f.n) {
            uint2 next;
            const FeatTerms v = feature_one<DT>(f, hilbert, og, i, p, bad, zero_q, next);
            if (last >= 0) f.cell[last] = ks;
            ks = next;
            last = i;
            acc.add(v);
        }
    }
    if (last >= 0) f.cell[last] = ks;
    if (!isfinite(bad)) set_status(f.status, kEnonfinite);
    if (zero_q) set_status(f.status, kEinval);
#pragma unroll
    for (int k = 0; k < kFeatSums; ++k) red[k * kFeatRedRow + t] = acc.s[k];
    __syncthreads();
    feature_block_sums(red, f.partials);
}

// Small scenes: the eight primitives that a thread of k_features would take
// one after the other (n is at most 8 x 256 x G) are taken by four threads,
// two each; their terms meet in shared memory and are added in the same order,
// so the sums have the same bits.  One CTA of 1,024 threads fills an SM's
// registers, so this is for scenes of at most one such block per SM.  10k
// primitives: 17 against 22 us; 150k: 18 against 24 us (events around the
// launch included, about 4 us).
constexpr int kFeatSmallThreads = 1024;

template <int DT>
__global__ void __launch_bounds__(kFeatSmallThreads, 1) k_features_small(FeatureArgs<DT> f)
{
    after(pdl_wait(), f.grid);  // the rows are older than the kernel before this one
    constexpr int kGroups = kFeatSmallThreads / kFeatCol;
    __shared__ float val[5][kFeatCols][kFeatCol];  // y, alpha, gem, m_gem, m_col
    __shared__ __align__(4) uint16_t hilbert[24 * 64];
    load_hilbert(hilbert);
    const OrderGrid og = *f.grid;
    __syncthreads();
    const int t = threadIdx.x % kFeatCol, grp = threadIdx.x / kFeatCol;
    const int64_t first = (int64_t)blockIdx.x * kFeatCol + t, step = (int64_t)gridDim.x * kFeatCol;
    float bad = 0.f;
    bool zero_q = false;
    uint2 ks[kFeatCols / kGroups];
#pragma unroll
    for (int u = 0; u < kFeatCols / kGroups; ++u) {
        const int c = u * kGroups + grp;
        const int64_t i = first + c * step;
        if (i < f.n) {
            const FeatTerms v = feature_one<DT>(f, hilbert, og, i, load_rows<DT>(f, i), bad, zero_q, ks[u]);
            val[0][c][t] = v.y;
            val[1][c][t] = v.alpha;
            val[2][c][t] = v.gem;
            val[3][c][t] = v.mg;
            val[4][c][t] = v.mc;
        }
    }
#pragma unroll
    for (int u = 0; u < kFeatCols / kGroups; ++u) {
        const int64_t i = first + (u * kGroups + grp) * step;
        if (i < f.n) f.cell[i] = ks[u];
    }
    if (!isfinite(bad)) set_status(f.status, kEnonfinite);
    if (zero_q) set_status(f.status, kEinval);
    __syncthreads();
    // the sums, dealt to the four groups
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int c = 0; c < kFeatCols; ++c) {
        if (first + c * step >= f.n) break;
        if (grp == 0) {
            const float y = val[0][c][t];
            s0 += y;
            s1 = fmaf(y, y, s1);
        } else if (grp == 1) {
            const float al = val[1][c][t];
            s0 = fmaf(al, 1.f - al, s0);
            s1 += al;
        } else if (grp == 2) {
            s0 += val[2][c][t];
            s1 += val[3][c][t];
        } else {
            s0 += val[4][c][t];
        }
    }
    __syncthreads();
    float *red = &val[0][0][0];
    const int k0 = grp == 0 ? 0 : (grp == 1 ? 2 : (grp == 2 ? 3 : 5)), k1 = grp == 0 ? 1 : (grp == 1 ? 6 : 4);
    red[k0 * kFeatRedRow + t] = s0;
    if (grp < 3) red[k1 * kFeatRedRow + t] = s1;
    __syncthreads();
    feature_block_sums(red, f.partials);
}

// Blocks of the sums: eight primitives a thread or more, a single wave of 4
// CTAs of k_features on each of 152 SMs; it depends only on n, so the
// per-block sums, and the scene constants, do too.
int feature_blocks(int64_t n)
{
    int64_t b = (n + (int64_t)kFeatCol * kFeatCols - 1) / ((int64_t)kFeatCol * kFeatCols);
    if (b < 1) b = 1;
    if (b > 608) b = 608;
    return (int)b;
}

template <int DT>
static cudaError_t launch_features_t(const FeatureLaunch &l, int num_sms, const Chain &s)
{
    FeatureArgs<DT> f{l.pos, AttrRows<DT>(l.attr, l.stride), l.stride, l.n, l.eta, l.luma[0], l.luma[1], l.luma[2], l.recs,
                      l.partials, l.grid, l.cell_bits, l.cell, l.counts, l.status};
    const int nb = feature_blocks(l.n);
    if (nb <= num_sms && l.n <= (int64_t)nb * kFeatCol * kFeatCols)
        return launch_chained(k_features_small<DT>, nb, kFeatSmallThreads, 0, s, f);
    if constexpr (DT != REFINE_F32) {
        using Rows = RowTile<DT, kFeatCol>;
        static_assert(Rows::kBytes + 12 * 1024 < 48 * 1024, "no opt-in shared memory");
        if (l.stride % 8 == 0)
            return launch_chained(k_features_bulk<DT, true>, nb, kFeatCol, Rows::kBytes, s, f,
                                  Rows(l.pos, l.attr, l.stride, Rows::whole_chunks(l.n)));
        return launch_chained(k_features_bulk<DT, false>, nb, kFeatCol, Rows::kBytes, s, f,
                              Rows(l.pos, l.attr, l.stride, l.n));
    } else {
        return launch_chained(k_features<DT>, nb, kFeatCol, 0, s, f);
    }
}

cudaError_t launch_features(const FeatureLaunch &f, int dtype, int num_sms, const Chain &s)
{
    if (dtype == REFINE_BF16) return launch_features_t<REFINE_BF16>(f, num_sms, s);
    if (dtype == REFINE_BF16S) return launch_features_t<REFINE_BF16S>(f, num_sms, s);
    return launch_features_t<REFINE_F32>(f, num_sms, s);
}

// Eq. (features) -> Eq. 18 -> Eq. 19 in double, by one block (every thread
// calls it), from the feature pass's block sums.  The scalar tail runs in
// three warps side by side (one attribute each, FP64 being the slow part).
__device__ void finalize_features(const SceneTail &f)
{
    // each sum k is reduced by one warp over the block partials in a fixed
    // order (lane-strided, then a shuffle tree) in float-float, whichever
    // warp it is, and converted to double once
    __shared__ double red[kFeatSums];
    __shared__ double lam_t[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < kFeatSums) {
        FF v = {0.f, 0.f};
#pragma unroll 4
        for (int b = lane; b < f.nblocks; b += 32) {
            const float2 q = __ldg(f.partials + (int64_t)b * kFeatSums + warp);
            v = ff_add(v, FF{q.x, q.y});
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            v = ff_add(v, FF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)});
        if (lane == 0) red[warp] = ff_to_double(v);
    }
    __syncthreads();
    const int t = warp;  // attribute: gem, col, opa
    const double N = (double)f.n;
    if (lane == 0 && t < 3) {
        double lt;
        if (t == 0) {
            lt = log(red[3] / N + (double)f.p.eta) / f.p.e_ln_gem;
        } else if (t == 1) {
            const double ybar = red[0] / N;
            double fc = red[1] / N - ybar * ybar;
            if (fc < 0.0) fc = 0.0;
            lt = fc / f.p.e_col;
            f.stats->F_col = fc;
        } else {
            lt = (red[2] / N) / f.p.e_opa;
        }
        if (!(lt > 0.0)) lt = 0.0;
        lam_t[t] = lt;
    }
    __syncthreads();
    if (lane != 0 || t >= 3) return;  // no barrier follows
    const double tot = (lam_t[0] + lam_t[1]) + lam_t[2];
    const double lambda = ((f.p.flags & REFINE_FLAG_EQUAL_LAMBDA) || tot == 0.0) ? 1.0 / 3.0 : lam_t[t] / tot;
    const double mean_m = red[4 + t] / N;
    double kap = lambda;
    if (f.p.flags & REFINE_FLAG_NORM_ATTR) kap = mean_m > 0.0 ? lambda / mean_m : 0.0;
    f.consts->kappa[t] = (float)kap;
    f.stats->lambda_t[t] = lam_t[t];
    f.stats->lambda[t] = lambda;
    f.stats->mean_m[t] = mean_m;
    if (t == 0) {
        f.stats->F_opa = red[2] / N;
        f.stats->F_gem = red[3] / N;
    }
}

// Exclusive scan of the cell counts: local offsets within blocks of
// kScanCells cells (4 consecutive cells per thread, one 16-byte load), then
// the last block turns the block totals into block offsets, so cell c
// starts at bsum[c / kScanCells] + off_local[c].
__device__ __forceinline__ unsigned block_excl_scan(unsigned v, unsigned *wsum)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned x = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += x;
    }
    if (lane == 31) wsum[warp] = s;
    __syncthreads();
    if (warp == 0) {
        unsigned w = wsum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned x = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += x;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    const unsigned r = s - v + (warp > 0 ? wsum[warp - 1] : 0u);
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kScanThreads) k_cell_scan(const unsigned *__restrict__ counts,
                                                            unsigned *__restrict__ off_local,
                                                            unsigned *bsum, unsigned *done)
{
    after(pdl_wait(), counts);
    const int nblocks = gridDim.x;
    __shared__ unsigned wsum[32];
    __shared__ unsigned is_last, carry;
    const int64_t c4 = (int64_t)blockIdx.x * kScanThreads + threadIdx.x;  // 4 cells from 4 * c4
    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(counts) + c4);
    const unsigned tot = v.x + v.y + v.z + v.w;
    const unsigned ex = block_excl_scan(tot, wsum);
    reinterpret_cast<uint4 *>(off_local)[c4] = make_uint4(ex, ex + v.x, ex + v.x + v.y, ex + v.x + v.y + v.z);
    if (threadIdx.x == kScanThreads - 1) bsum[blockIdx.x] = ex + tot;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = (int)atomicAdd(done, 1u) == nblocks - 1;
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    if (threadIdx.x == 0) carry = 0u;
    __syncthreads();
    for (int b0 = 0; b0 < nblocks; b0 += kScanThreads) {
        const int bi = b0 + threadIdx.x;
        const unsigned b = bi < nblocks ? __ldcg(bsum + bi) : 0u;
        const unsigned bex = block_excl_scan(b, wsum) + carry;
        __syncthreads();
        if (bi < nblocks) bsum[bi] = bex;
        if (threadIdx.x == kScanThreads - 1) carry = bex + b;
        __syncthreads();
    }
}

cudaError_t launch_cell_scan(unsigned *counts, unsigned *off_local, unsigned *bsum, unsigned *done, int cell_bits,
                             const Chain &s)
{
    return launch_chained(k_cell_scan, order_keys(cell_bits) / kScanCells, kScanThreads, 0, s, counts, off_local, bsum, done);
}

constexpr int kSortU = 4;  // primitives in flight per thread

static int sort_grid(int num_sms, int64_t n)
{
    int64_t g = (n + 255) / 256;
    if (g > (int64_t)num_sms * 8) g = (int64_t)num_sms * 8;
    if (g < 1) g = 1;
    return (int)g;
}

// Primitive j goes to the start of its cell (block offset + offset within
// the block) plus the slot that its count atomic returned.  Block 0 forms the
// scene constants meanwhile (finalize_features): nothing before the score
// kernel's last step needs them, and their FP64 chain at the end of the
// feature pass held up everything after it.
__global__ void __launch_bounds__(256) k_cell_scatter(const uint2 *__restrict__ cell, int64_t n,
                                                      const unsigned *__restrict__ off_local,
                                                      const unsigned *__restrict__ boff, uint32_t *__restrict__ perm,
                                                      SceneTail tail)
{
    const int64_t zero = pdl_wait();
    after(zero, off_local);  // (the rest is older than the kernel before this one)
    after(zero, boff);
    if (blockIdx.x == 0) {
        finalize_features(tail);
        return;
    }
    const int64_t step = (int64_t)(gridDim.x - 1) * blockDim.x;
    for (int64_t i = (int64_t)(blockIdx.x - 1) * blockDim.x + threadIdx.x; i < n; i += kSortU * step) {
        uint2 c[kSortU];
#pragma unroll
        for (int u = 0; u < kSortU; ++u) {
            const int64_t j = i + u * step;
            c[u] = j < n ? __ldg(cell + j) : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < kSortU; ++u) {
            const int64_t j = i + u * step;
            if (j < n) perm[__ldg(boff + c[u].x / kScanCells) + __ldg(off_local + c[u].x) + c[u].y] = (uint32_t)j;
        }
    }
}

cudaError_t launch_cell_scatter(const uint2 *cell, int64_t n, const unsigned *off_local, const unsigned *bsum,
                                uint32_t *perm, const SceneTail &tail, int num_sms, const Chain &s)
{
    return launch_chained(k_cell_scatter, sort_grid(num_sms, n) + 1, 256, 0, s, cell, n, off_local, bsum, perm, tail);
}

}  // namespace refine
