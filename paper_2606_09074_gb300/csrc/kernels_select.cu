// Ratio pruning (Sec. 3.3): radix select of the n_keep-th largest score with
// an index tie-break, keep-mask construction, and stable compaction.
#include <cooperative_groups.h>

#include "internal.h"

namespace refine {

namespace cg = cooperative_groups;

// Radix digits from the most significant end: 11, 11 and 10 bits.
__host__ __device__ constexpr int pass_shift(int p) { return p == 0 ? 21 : (p == 1 ? 10 : 0); }
__host__ __device__ constexpr int pass_width(int p) { return p == 2 ? 10 : 11; }

constexpr int kSelThreads = 512;

// Inclusive suffix sum over the block (thread t receives the sum of the
// values of threads t..blockDim-1), blockDim == kSelThreads.
__device__ unsigned int block_suffix_sum(unsigned int v, unsigned int *wsum)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned int s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned int x = __shfl_down_sync(0xffffffffu, s, o);
        if (lane + o < 32) s += x;
    }
    if (lane == 0) wsum[warp] = s;
    __syncthreads();
    if (warp == 0) {
        unsigned int w = lane < kSelThreads / 32 ? wsum[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned int x = __shfl_down_sync(0xffffffffu, w, o);
            if (lane + o < 32) w += x;
        }
        if (lane < kSelThreads / 32) wsum[lane] = w;  // inclusive suffix over warps
    }
    __syncthreads();
    unsigned int after = (warp + 1 < kSelThreads / 32) ? wsum[warp + 1] : 0u;
    unsigned int r = s + after;
    __syncthreads();
    return r;
}

// Inclusive prefix sum over the block.
__device__ unsigned long long block_prefix_sum(unsigned long long v, unsigned long long *wsum)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    unsigned long long s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long x = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += x;
    }
    if (lane == 31) wsum[warp] = s;
    __syncthreads();
    if (warp == 0) {
        unsigned long long w = lane < nw ? wsum[lane] : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long x = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += x;
        }
        if (lane < nw) wsum[lane] = w;
    }
    __syncthreads();
    unsigned long long r = s + (warp > 0 ? wsum[warp - 1] : 0ull);
    __syncthreads();
    return r;
}

// Adds one count for digit d of the lanes with `match` to the histogram.
// Shared-memory atomics take equal addresses of a warp one by one, which is
// cheap for a few, so only the commonest case of many is grouped: the lanes
// that share the first matching lane's digit (zeros, and the few exponents
// that most scores have) go in one add.  Every lane of the warp calls it.
__device__ __forceinline__ void hist_add(unsigned *h, unsigned d, bool match)
{
    const unsigned any = __ballot_sync(0xffffffffu, match);
    if (!any) return;
    const int lead = __ffs(any) - 1;
    const unsigned d0 = __shfl_sync(0xffffffffu, d, lead);
    const unsigned same = __ballot_sync(0xffffffffu, match && d == d0);
    if ((int)(threadIdx.x & 31) == lead)
        atomicAdd(&h[d0], (unsigned)__popc(same));
    else if (match && d != d0)
        atomicAdd(&h[d], 1u);
}

// One histogram pass over the keys that match the digits decided so far.
// The last CTA to finish chooses the digit of the n_keep-th largest key.
// The scores are in L2 after the score kernel; what counts is loads in flight
// (kSelU 16-byte loads a thread) and the histogram adds: 53 against 60 us a
// selection of 3.5M scores, 36 against 40 us of 1M, with one load a thread and
// every digit grouped by a match of the whole warp.
constexpr int kSelU = 4;

template <int PASS, bool VEC>
__global__ void __launch_bounds__(kSelThreads) k_select_pass(const float *__restrict__ scores, int64_t n,
                                                             uint32_t n_keep, SelState *st, int *status)
{
    constexpr int SHIFT = pass_shift(PASS), WIDTH = pass_width(PASS), NB = 1 << WIDTH;
    __shared__ unsigned int h[2048];
    __shared__ unsigned int wsum[32];
    __shared__ unsigned int is_last;
    for (int b = threadIdx.x; b < NB; b += blockDim.x) h[b] = 0u;
    after(pdl_wait(), scores);
    __syncthreads();
    const unsigned int prefix = PASS == 0 ? 0u : st->prefix;
    bool bad = false;
    // Every lane of a warp runs the same iterations (warp-uniform bounds), so
    // the full-mask votes see a converged warp; `valid` masks lanes.
    auto add = [&](float f, bool valid) {
        if (PASS == 0) bad |= valid && isnan(f);
        const uint32_t k = score_key(f);
        hist_add(h, (k >> SHIFT) & (NB - 1), valid && (PASS == 0 ? true : ((k >> (SHIFT + WIDTH)) == prefix)));
    };
    const int lane = threadIdx.x & 31;
    const int64_t wbase = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
    const int64_t nthr = (int64_t)gridDim.x * blockDim.x;
    int64_t done_to = 0;
    if (VEC) {
        const int64_t n4 = n / 4;
        const float4 *s4 = reinterpret_cast<const float4 *>(scores);
        for (int64_t i0 = wbase; i0 < n4; i0 += kSelU * nthr) {
            float4 q[kSelU];
#pragma unroll
            for (int u = 0; u < kSelU; ++u) {
                const int64_t i = i0 + u * nthr + lane;
                q[u] = i < n4 ? __ldg(s4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < kSelU; ++u) {
                if (i0 + u * nthr >= n4) break;  // uniform in the warp
                const bool valid = i0 + u * nthr + lane < n4;
                add(q[u].x, valid); add(q[u].y, valid); add(q[u].z, valid); add(q[u].w, valid);
            }
        }
        done_to = n4 * 4;
    }
    for (int64_t i0 = done_to + wbase; i0 < n; i0 += nthr) {
        const int64_t i = i0 + lane;
        const bool valid = i < n;
        add(valid ? __ldg(scores + i) : 0.f, valid);
    }
    if (PASS == 0 && bad) set_status(status, kEnonfinite);
    __syncthreads();
    for (int b = threadIdx.x; b < NB; b += blockDim.x)
        if (h[b]) atomicAdd(&st->hist[b], h[b]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = (atomicAdd(&st->done, 1u) == gridDim.x - 1);
    __syncthreads();
    if (!is_last) return;
    __threadfence();

    // Choose the bucket: thread t owns bins [t*PER, t*PER + PER).
    constexpr int PER = NB / kSelThreads;
    unsigned int cnt[PER], loc = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        cnt[k] = __ldcg(&st->hist[threadIdx.x * PER + k]);  // from L2, where the atomics were
        loc += cnt[k];
    }
    const unsigned int remaining = PASS == 0 ? n_keep : st->remaining;
    const unsigned int incl = block_suffix_sum(loc, wsum);  // bins >= my first bin
    const unsigned int excl = incl - loc;                   // bins above my range
    if (excl < remaining && remaining <= incl) {
        unsigned int above = excl;
        for (int k = PER - 1; k >= 0; --k) {
            if (above + cnt[k] >= remaining) {
                const unsigned int digit = threadIdx.x * PER + k;
                const unsigned int rem = remaining - above;
                st->remaining = rem;
                st->prefix = (prefix << WIDTH) | digit;
                if (PASS == 2) {
                    st->kstar = (prefix << WIDTH) | digit;
                    st->need_ties = cnt[k] > rem ? 1u : 0u;
                    st->idx_cut = n;  // refined by k_select_ties when needed
                }
                break;
            }
            above += cnt[k];
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) st->hist[threadIdx.x * PER + k] = 0u;
    if (threadIdx.x == 0) st->done = 0u;
}

int select_grid(int num_sms, int64_t n)
{
    int64_t g = (n + (int64_t)kSelThreads * 8 - 1) / ((int64_t)kSelThreads * 8);
    if (g > 2 * num_sms) g = 2 * num_sms;
    if (g < 1) g = 1;
    return (int)g;
}

template <int PASS>
static cudaError_t launch_pass_t(const float *scores, int64_t n, uint32_t n_keep, SelState *st,
                                 bool vec, int grid, int *status, const Chain &s)
{
    if (vec) return launch_chained(k_select_pass<PASS, true>, grid, kSelThreads, 0, s, scores, n, n_keep, st, status);
    return launch_chained(k_select_pass<PASS, false>, grid, kSelThreads, 0, s, scores, n, n_keep, st, status);
}

cudaError_t launch_select_pass(int pass, const float *scores, int64_t n, uint32_t n_keep,
                               SelState *st, bool vec, int grid, int *status, const Chain &s)
{
    if (pass == 0) return launch_pass_t<0>(scores, n, n_keep, st, vec, grid, status, s);
    if (pass == 1) return launch_pass_t<1>(scores, n, n_keep, st, vec, grid, status, s);
    return launch_pass_t<2>(scores, n, n_keep, st, vec, grid, status, s);
}

// Index tie-break: when more keys equal k* than remain to be kept, find the
// index of the `remaining`-th such key in index order.  Segments of kTieSeg
// elements are counted; the last CTA locates the segment and the element.
__global__ void __launch_bounds__(kSelThreads) k_select_ties(const float *__restrict__ scores, int64_t n,
                                                             SelState *st, unsigned *seg_cnt)
{
    after(pdl_wait(), scores);
    if (!st->need_ties) return;
    __shared__ unsigned long long wsum[32];
    __shared__ unsigned int is_last;
    __shared__ long long found_seg;
    __shared__ unsigned long long seg_base;
    const uint32_t kstar = st->kstar;
    const int64_t nseg = (n + kTieSeg - 1) / kTieSeg;
    for (int64_t sg = blockIdx.x; sg < nseg; sg += gridDim.x) {
        unsigned int c = 0;
        const int64_t e1 = min(n, (sg + 1) * (int64_t)kTieSeg);
        for (int64_t i = sg * (int64_t)kTieSeg + threadIdx.x; i < e1; i += blockDim.x)
            c += score_key(__ldg(scores + i)) == kstar;
        for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
        __shared__ unsigned int red[kSelThreads / 32];
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned int t = 0;
            for (int w = 0; w < kSelThreads / 32; ++w) t += red[w];
            seg_cnt[sg] = t;
        }
        __syncthreads();
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = (atomicAdd(&st->done, 1u) == gridDim.x - 1);
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    const unsigned long long target = st->remaining;  // 1-based rank among equal keys
    if (threadIdx.x == 0) found_seg = -1;
    __syncthreads();
    unsigned long long run = 0;
    for (int64_t c0 = 0; c0 < nseg; c0 += blockDim.x) {
        const int64_t sg = c0 + threadIdx.x;
        const unsigned long long v = sg < nseg ? atomicAdd(&seg_cnt[sg], 0u) : 0ull;
        const unsigned long long incl = block_prefix_sum(v, wsum) + run;
        if (sg < nseg && incl - v < target && target <= incl) {
            found_seg = sg;
            seg_base = incl - v;
        }
        __syncthreads();
        if (found_seg >= 0) break;
        // the running total is the inclusive sum of the chunk's last thread
        __shared__ unsigned long long chunk_end;
        if (threadIdx.x == blockDim.x - 1) chunk_end = incl;
        __syncthreads();
        run = chunk_end;
        __syncthreads();
    }
    const int64_t sg = found_seg;
    if (sg >= 0) {
        unsigned long long base = seg_base;
        const int64_t e1 = min(n, (sg + 1) * (int64_t)kTieSeg);
        for (int64_t i0 = sg * (int64_t)kTieSeg; i0 < e1; i0 += blockDim.x) {
            const int64_t i = i0 + threadIdx.x;
            const unsigned long long eq = (i < e1 && score_key(__ldg(scores + i)) == kstar) ? 1ull : 0ull;
            const unsigned long long incl = block_prefix_sum(eq, wsum) + base;
            if (eq && incl == target) st->idx_cut = i;
            __shared__ unsigned long long cend;
            if (threadIdx.x == blockDim.x - 1) cend = incl;
            __syncthreads();
            base = cend;
            __syncthreads();
            if (base >= target) break;
        }
    }
    if (threadIdx.x == 0) st->done = 0u;
}

cudaError_t launch_select_ties(const float *scores, int64_t n, SelState *st, unsigned *seg_cnt,
                               int grid, const Chain &s)
{
    return launch_chained(k_select_ties, grid, kSelThreads, 0, s, scores, n, st, seg_cnt);
}

// Keep mask: a warp builds kMaskWords consecutive 32-element words per
// step, their loads issued together.
constexpr int kMaskWords = 8;

__global__ void k_select_mask(const float *__restrict__ scores, int64_t n, const SelState *st,
                              uint32_t *__restrict__ mask)
{
    const int64_t zero = pdl_wait();
    after(zero, scores);
    after(zero, st);
    const uint32_t kstar = st->kstar;
    const long long cut = st->idx_cut;
    const int64_t words = (n + 31) / 32;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w0 = warp0 * kMaskWords; w0 < words; w0 += nwarps * kMaskWords) {
        float v[kMaskWords];
#pragma unroll
        for (int u = 0; u < kMaskWords; ++u) {
            const int64_t i = (w0 + u) * 32 + lane;
            v[u] = i < n ? __ldg(scores + i) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kMaskWords; ++u) {
            const int64_t i = (w0 + u) * 32 + lane;
            const uint32_t k = score_key(v[u]);
            const bool keep = i < n && (k > kstar || (k == kstar && i <= cut));
            const uint32_t word = __ballot_sync(0xffffffffu, keep);
            if (lane == 0 && w0 + u < words) mask[w0 + u] = word;
        }
    }
}

cudaError_t launch_select_mask(const float *scores, int64_t n, const SelState *st, uint32_t *mask,
                               int num_sms, const Chain &s)
{
    // one step of every warp, up to 8 CTAs of 8 warps per SM
    int64_t g = ((n + 31) / 32 + 8 * kMaskWords - 1) / (8 * kMaskWords);
    if (g > (int64_t)num_sms * 8) g = (int64_t)num_sms * 8;
    if (g < 1) g = 1;
    return launch_chained(k_select_mask, (int)g, 256, 0, s, scores, n, st, mask);
}

// ---------------------------------------------------------------------
// The whole selection in one launch of one thread-block cluster, for up to
// kSelClusterMax scores: CTA r holds the keys of its range in shared memory,
// so the scores are read once.  Three digits as above: each CTA counts its
// keys, the cluster meets at its (hardware) barrier, and every CTA adds all
// histograms through distributed shared memory and picks the same digit.
// Among keys equal to k* the first in index order are kept: the CTAs exchange
// their counts of them and each cuts its own range.  Then each writes the mask
// words of its range.
//
// What it saves is launches: six stream operations become one.  The cluster
// has 1, 2, 4 or 8 CTAs, 6k keys each before the next size is taken (10k scores
// take 8.0 us with 2 CTAs, 10.3 with 1, 11.4 with 8; 24k 10.1 with 4, 12.8 with
// 2, 12.2 with 8).  Per selection, chained: 1k scores 5.6, 10k 8.7, 50k 14.8,
// 100k 19.0, 131k 21.2 us, against the five kernels and a memset of the other
// form, a chain of latencies that takes 22.5-23 us from 131k to 400k scores.
// Not chained, with a memset before: 100k 25, 200k 33, 262k 37 us, against 33 us.
// In a batch's graph, which saves five nodes: alone, 150k as fast, 190k 4 and
// 250k 8 us slower; 8 scenes of 150k or 190k 6 us of 180 faster, of 250k 2, 24 of
// 250k 5 us of 740 slower.  In the queue, whose scorer issues every launch: three
// jobs of 200k at once 785 against 862 us, eight 1,650 against 1,690, of 250k 2,130
// against 2,180.  Hence the limits, kSelClusterChained and kSelClusterMax (batch
// and queue).
// ---------------------------------------------------------------------
constexpr int kClThreads = 1024;
constexpr int kClKeys = 32 * 1024;  // keys of a CTA at most (128 KB)
constexpr int kClMaxCtas = 8;
constexpr int kClFill = 6 * 1024;  // keys per CTA at which a larger cluster is taken
constexpr int kClLoads = 6;         // loads in flight per thread
static_assert(kSelClusterMax == (int64_t)kClKeys * kClMaxCtas, "cluster selection limit");

__global__ void __launch_bounds__(kClThreads) k_select_cluster(const float *__restrict__ scores, int n, int per,
                                                               uint32_t n_keep, SelState *st, uint32_t *__restrict__ mask,
                                                               int *status)
{
    extern __shared__ uint32_t keys[];
    __shared__ unsigned hist[3][2048];
    __shared__ unsigned wsum[kClThreads / 32];
    __shared__ unsigned pick[3], equal;
    cg::cluster_group cl = cg::this_cluster();
    const int ctas = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = rank * per, m = max(0, min(per, n - i0));  // per is a multiple of 32
    for (int b = threadIdx.x; b < 3 * 2048; b += kClThreads) (&hist[0][0])[b] = 0u;
    after(pdl_wait(), scores);
    __syncthreads();
    bool bad = false;
    for (int j0 = warp * 32; j0 < m; j0 += kClLoads * kClThreads) {
        float f[kClLoads];
#pragma unroll
        for (int u = 0; u < kClLoads; ++u) {
            const int j = j0 + u * kClThreads + lane;
            f[u] = j < m ? __ldg(scores + i0 + j) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kClLoads; ++u) {
            const int j = j0 + u * kClThreads + lane;
            if (j - lane >= m) break;  // uniform in the warp
            bad |= isnan(f[u]);
            const uint32_t k = score_key(f[u]);
            if (j < m) keys[j] = k;
            hist_add(hist[0], k >> pass_shift(0), j < m);
        }
    }
    if (bad) set_status(status, kEnonfinite);
    unsigned prefix = 0u, remaining = n_keep, count = 0u;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        if (p > 0) {
            __syncthreads();
            for (int j0 = warp * 32; j0 < m; j0 += kClThreads) {
                const int j = j0 + lane;
                const uint32_t k = j < m ? keys[j] : 0u;
                hist_add(hist[p], (k >> pass_shift(p)) & ((1u << pass_width(p)) - 1u),
                         j < m && (k >> (pass_shift(p) + pass_width(p))) == prefix);
            }
        }
        cl.sync();
        // thread t owns bins 2t and 2t + 1; suffix sums over the block
        uint2 c = make_uint2(0u, 0u);
        for (int r = 0; r < ctas; ++r) {
            const uint2 q = *reinterpret_cast<const uint2 *>(cl.map_shared_rank(&hist[p][2 * threadIdx.x], r));
            c.x += q.x;
            c.y += q.y;
        }
        unsigned s = c.x + c.y;
        const unsigned own = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned x = __shfl_down_sync(0xffffffffu, s, o);
            if (lane + o < 32) s += x;
        }
        if (lane == 0) wsum[warp] = s;
        __syncthreads();
        unsigned w = lane > warp ? wsum[lane] : 0u;  // the warps above
        w = __reduce_add_sync(0xffffffffu, w);
        const unsigned excl = s - own + w;  // keys in bins above mine
        if (excl < remaining && remaining <= excl + own) {
            const bool hi = excl + c.y >= remaining;
            const unsigned above = hi ? excl : excl + c.y;
            pick[0] = 2u * threadIdx.x + (hi ? 1u : 0u);
            pick[1] = remaining - above;
            pick[2] = hi ? c.y : c.x;
        }
        __syncthreads();
        prefix = (prefix << pass_width(p)) | pick[0];
        remaining = pick[1];
        count = pick[2];
        __syncthreads();
    }
    const uint32_t kstar = prefix;
    int cut = m;  // keys equal to k* are kept below this position of the range
    if (count > remaining) {  // the same in every CTA
        // each thread counts a run of positions of the range
        const int run = (m + kClThreads - 1) / kClThreads;
        const int a = min(m, (int)threadIdx.x * run), b = min(m, a + run);
        unsigned e = 0u;
        for (int j = a; j < b; ++j) e += keys[j] == kstar;
        unsigned s = e;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned x = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += x;
        }
        if (lane == 31) wsum[warp] = s;
        __syncthreads();
        const unsigned below = __reduce_add_sync(0xffffffffu, lane < warp ? wsum[lane] : 0u);
        const unsigned before_me = below + s - e;
        if (threadIdx.x == kClThreads - 1) equal = below + s;
        if (threadIdx.x == 0) pick[0] = (unsigned)m;
        cl.sync();
        unsigned before = 0u;
        for (int r = 0; r < rank; ++r) before += *cl.map_shared_rank(&equal, r);
        // position after the last kept one of this range (m when all are kept)
        const unsigned left = remaining > before ? remaining - before : 0u;
        if (left == 0u) {
            if (threadIdx.x == 0) pick[0] = 0u;
        } else if (before_me < left && left <= before_me + e) {
            unsigned seen = before_me;
            for (int j = a; j < b; ++j)
                if (keys[j] == kstar && ++seen == left) {
                    pick[0] = (unsigned)(j + 1);
                    break;
                }
        }
        __syncthreads();
        cut = (int)pick[0];
    }
    for (int j0 = warp * 32; j0 < m; j0 += kClThreads) {
        const int j = j0 + lane;
        const uint32_t k = j < m ? keys[j] : 0u;
        const uint32_t word = __ballot_sync(0xffffffffu, j < m && (k > kstar || (k == kstar && j < cut)));
        if (lane == 0) mask[(i0 + j0) >> 5] = word;
    }
    if (rank == 0 && threadIdx.x == 0) st->kstar = kstar;
    cl.sync();  // no CTA leaves while another may read its shared memory
}

cudaError_t launch_select_cluster(const float *scores, int64_t n, uint32_t n_keep, SelState *st, uint32_t *mask,
                                  int *status, const Chain &s)
{
    int ctas = 1;
    while (ctas < kClMaxCtas && n > (int64_t)kClFill * ctas) ctas *= 2;
    const int per = (int)(((n + ctas - 1) / ctas + 31) / 32 * 32);
    const size_t smem = sizeof(uint32_t) * (size_t)per;
    if (smem + 3 * 2048 * sizeof(unsigned) + 1024 > 48 * 1024) {
        // one constant for every launch: a smaller value set for one thread's
        // launch would refuse another's larger one
        const cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(&k_select_cluster),
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(sizeof(uint32_t) * kClKeys));
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s.s;
    cudaLaunchAttribute at[2]{};
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = s.on ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, k_select_cluster, scores, (int)n, per, n_keep, st, mask, status);
}

__global__ void k_mask_fill(uint32_t *mask, int64_t n)
{
    after(pdl_wait(), mask);
    const int64_t words = (n + 31) / 32;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < words;
         w += (int64_t)gridDim.x * blockDim.x) {
        const int64_t rem = n - w * 32;
        mask[w] = rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u);
    }
}

cudaError_t launch_mask_fill(uint32_t *mask, int64_t n, const Chain &s)
{
    int64_t words = (n + 31) / 32;
    int grid = (int)((words + 255) / 256);
    if (grid > 1024) grid = 1024;
    if (grid < 1) grid = 1;
    return launch_chained(k_mask_fill, grid, 256, 0, s, mask, n);
}

// ---------------------------------------------------------------------
// Compaction, pass 1.  Segment s covers elements [s*kCmpSeg, (s+1)*kCmpSeg)
// (8 mask words).
//
// Up to kCmpMaxBlocks blocks of kCmpBlockSegs segments (k_compact_local): a
// block counts its segments and leaves their offsets within it and its total;
// every CTA of the scatter adds up the totals.  No CTA waits for the others
// and nothing needs clearing: 6 against 18 us (3.5M) and 10 us (1M).
// Larger scenes (k_compact_count): the last CTA turns all the counts into
// offsets.
// ---------------------------------------------------------------------
__global__ void __launch_bounds__(kCmpBlockSegs) k_compact_local(const uint32_t *__restrict__ mask, int64_t n,
                                                                 unsigned *__restrict__ local,
                                                                 unsigned *__restrict__ totals)
{
    constexpr int kWords = kCmpSeg / 32;
    static_assert(kWords == 8, "a segment is two 16-byte loads");
    __shared__ unsigned wsum[kCmpBlockSegs / 32];
    after(pdl_wait(), mask);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t sg = (int64_t)blockIdx.x * kCmpBlockSegs + threadIdx.x, nseg = (n + kCmpSeg - 1) / kCmpSeg;
    const int64_t words = (n + 31) / 32;
    unsigned c = 0u;
    if ((sg + 1) * kCmpSeg <= n && (reinterpret_cast<uintptr_t>(mask) & 15u) == 0) {
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(mask) + 2 * sg);
        const uint4 b = __ldg(reinterpret_cast<const uint4 *>(mask) + 2 * sg + 1);
        c = __popc(a.x) + __popc(a.y) + __popc(a.z) + __popc(a.w) + __popc(b.x) + __popc(b.y) + __popc(b.z) + __popc(b.w);
    } else {
#pragma unroll
        for (int k = 0; k < kWords; ++k) {
            const int64_t w = sg * kWords + k;
            if (w < words) {
                uint32_t word = __ldg(mask + w);
                const int64_t valid = n - w * 32;  // bits past n do not count
                if (valid < 32) word &= (1u << valid) - 1u;
                c += __popc(word);
            }
        }
    }
    unsigned s = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned x = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += x;
    }
    if (lane == 31) wsum[warp] = s;
    __syncthreads();
    unsigned below = 0u;
#pragma unroll
    for (int w = 0; w < kCmpBlockSegs / 32; ++w) below += w < warp ? wsum[w] : 0u;
    if (sg < nseg) local[sg] = below + s - c;
    if (threadIdx.x == kCmpBlockSegs - 1) totals[blockIdx.x] = below + s;
}

cudaError_t launch_compact_local(const uint32_t *mask, int64_t n, unsigned *local, unsigned *totals, const Chain &s)
{
    return launch_chained(k_compact_local, cmp_blocks(n), kCmpBlockSegs, 0, s, mask, n, local, totals);
}

constexpr int kCmpThreads = 1024;

__global__ void __launch_bounds__(kCmpThreads) k_compact_count(const uint32_t *__restrict__ mask, int64_t n,
                                                               unsigned *seg_cnt, unsigned long long *seg_off,
                                                               CmpState *cs, int64_t out_stride, int *status)
{
    __shared__ unsigned long long wsum[32];
    __shared__ unsigned int is_last;
    after(pdl_wait(), mask);
    const int64_t words = (n + 31) / 32;
    const int64_t nseg = (n + kCmpSeg - 1) / kCmpSeg;
    constexpr int kWords = kCmpSeg / 32;
    for (int64_t sg = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; sg < nseg;
         sg += (int64_t)gridDim.x * blockDim.x) {
        unsigned c = 0;
#pragma unroll
        for (int k = 0; k < kWords; ++k) {
            const int64_t w = sg * kWords + k;
            if (w < words) {
                uint32_t word = __ldg(mask + w);
                const int64_t valid = n - w * 32;  // bits past n do not count
                if (valid < 32) word &= (1u << valid) - 1u;
                c += __popc(word);
            }
        }
        seg_cnt[sg] = c;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = (atomicAdd(&cs->done, 1u) == gridDim.x - 1);
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    // thread t takes kCmpScanU consecutive segment counts per chunk (read
    // from L2, where the other blocks' counts are)
    constexpr int kCmpScanU = 4;
    unsigned long long run = 0;
    __shared__ unsigned long long chunk_end;
    for (int64_t c0 = 0; c0 < nseg; c0 += (int64_t)blockDim.x * kCmpScanU) {
        const int64_t sg0 = c0 + (int64_t)threadIdx.x * kCmpScanU;
        unsigned v[kCmpScanU];
        unsigned long long local = 0;
#pragma unroll
        for (int u = 0; u < kCmpScanU; ++u) {
            v[u] = sg0 + u < nseg ? __ldcg(seg_cnt + sg0 + u) : 0u;
            local += v[u];
        }
        const unsigned long long incl = block_prefix_sum(local, wsum) + run;
        unsigned long long o = incl - local;
#pragma unroll
        for (int u = 0; u < kCmpScanU; ++u) {
            if (sg0 + u < nseg) seg_off[sg0 + u] = o;
            o += v[u];
        }
        if (threadIdx.x == blockDim.x - 1) chunk_end = incl;
        __syncthreads();
        run = chunk_end;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        cs->total = (long long)run;
        cs->ok = run <= (unsigned long long)out_stride ? 1u : 0u;
        if (!cs->ok) set_status(status, kEinval);
        cs->done = 0u;
    }
}

cudaError_t launch_compact_count(const uint32_t *mask, int64_t n, unsigned *seg_cnt,
                                 unsigned long long *seg_off, CmpState *cs, int64_t out_stride,
                                 int grid, int *status, const Chain &s)
{
    return launch_chained(k_compact_count, grid, kCmpThreads, 0, s, mask, n, seg_cnt, seg_off, cs, out_stride, status);
}

}  // namespace refine
