// Compaction, pass 2: the scatter of every row of the kept primitives.
//
// One CTA of 8 warps takes a unit of consecutive primitives (128 with float32
// rows, 256 with bfloat16 rows) at a time.  The unit's span of each of the 59
// rows, 512 contiguous bytes (1 KB of a float32 row beside bfloat16 ones), is
// brought into shared memory by one bulk copy (cp.async.bulk) per row,
// completing on an mbarrier (RowTile); meanwhile the ranks
// of the kept primitives are inverted (output d comes from primitive src[d]).
// Then each warp takes every eighth row: 32 outputs are one shared-memory load
// and one contiguous store.  A unit is 31-34 KB, so 6 CTAs fit an SM, and while
// some wait for their unit others store theirs: about 190 KB an SM in flight
// without holding a register.
//
// Measured (the kernel alone, events around it): bfloat16 rows, 3.5M
// primitives at ratio 0.5 160 -> 107 us (6.2 TB/s); float32 rows 200 -> 199 us
// (3.5M, 6.3 TB/s) and 60 -> 55 us (1M at 0.66), against the form before, in
// which a warp loaded each row of a mask word into registers (16 float or 28
// bfloat16 rows at a time) and shuffled: 64-byte loads of bfloat16 rows, and
// registers, bounded what it had in flight.
#include "internal.h"
#include "rows.cuh"

namespace refine {

constexpr int kCmpWarps = 8;
constexpr int kCmpThreads = 32 * kCmpWarps;
constexpr int kCmpCtas = 6;  // per SM

// Primitives per unit.
__host__ __device__ constexpr int cmp_unit(int dtype) { return dtype == REFINE_F32 ? 128 : 256; }

template <int DT>
using CmpRows = RowTile<DT, cmp_unit(DT)>;

template <int DT>
__global__ void __launch_bounds__(kCmpThreads, kCmpCtas) k_compact(CmpRows<DT> in, int64_t n, const uint32_t *__restrict__ mask,
                                                         CmpOffsets off, char *__restrict__ out_pos,
                                                         char *__restrict__ out_attr, int64_t OS,
                                                         int32_t *__restrict__ out_idx, int *status)
{
    constexpr int UNIT = cmp_unit(DT), UW = UNIT / 32, SEGU = kCmpSeg / UNIT;
    extern __shared__ __align__(16) unsigned char tile[];
    __shared__ unsigned char src_of[UNIT];
    __shared__ unsigned blk_off[kCmpMaxBlocks];
    __shared__ unsigned wsum[kCmpWarps];
    __shared__ __align__(8) uint64_t bar;
    __shared__ int row_base[59];  // of each row in the tile, its misalignment included
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t units = (n + UNIT - 1) / UNIT, words = (n + 31) / 32;
    const int64_t zero = pdl_wait();
    after(zero, off.local);  // (the rows and the mask are older than the kernel before this one)
    after(zero, off.totals);
    after(zero, off.global);

    // Offsets of the blocks of segments from their totals (up to one total a
    // thread), and the kept count.
    if (off.blocks > 0) {
        static_assert(kCmpMaxBlocks == kCmpThreads, "one total per thread");
        const unsigned own = (int)threadIdx.x < off.blocks ? __ldg(off.totals + threadIdx.x) : 0u;
        unsigned s = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned x = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += x;
        }
        if (lane == 31) wsum[warp] = s;
        __syncthreads();
        unsigned below = 0u, total = 0u;
#pragma unroll
        for (int w = 0; w < kCmpWarps; ++w) {
            below += w < warp ? wsum[w] : 0u;
            total += wsum[w];
        }
        blk_off[threadIdx.x] = below + s - own;
        const bool ok = (int64_t)total <= OS;
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            off.state->total = (long long)total;
            if (!ok) set_status(status, kEinval);
        }
        if (!ok) return;
    } else if (!off.state->ok) {
        return;
    }
    if (threadIdx.x < 59)
        row_base[threadIdx.x] = CmpRows<DT>::place(threadIdx.x) + (int)in.mis(threadIdx.x);
    if (threadIdx.x == 0) mbar_init(&bar, 1);
    __syncthreads();

    uint32_t phase = 0;
    // word of the unit, bits past n cleared (lanes < UW of every warp)
    auto load_word = [&](int64_t u) {
        const int64_t w = u * UW + lane;
        uint32_t word = 0u;
        if (lane < UW && u < units && w < words) {
            word = __ldg(mask + w);
            const int64_t valid = n - w * 32;
            if (valid < 32) word &= (1u << valid) - 1u;
        }
        return word;
    };
    uint32_t next_word = load_word(blockIdx.x);
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        const uint32_t word = next_word;
        next_word = load_word(u + gridDim.x);
        const int kept = __reduce_add_sync(0xffffffffu, (unsigned)__popc(word));
        if (kept == 0) continue;  // the same in every thread
        const int64_t i0 = u * UNIT;
        const int count = (int)min((int64_t)UNIT, n - i0);
        in.template stage<kCmpWarps>(tile, i0, count, &bar);
        if (in.at_end(i0, n)) in.template rest<kCmpWarps>(tile, i0, count);
        // invert the ranks of the kept primitives
        {
            unsigned before = (unsigned)__popc(word);  // inclusive scan over the unit's words
#pragma unroll
            for (int o = 1; o < UW; o <<= 1) {
                const unsigned x = __shfl_up_sync(0xffffffffu, before, o);
                if (lane >= o) before += x;
            }
            before -= (unsigned)__popc(word);
            if (warp < UW) {
                const uint32_t mine = __shfl_sync(0xffffffffu, word, warp);
                const unsigned b = __shfl_sync(0xffffffffu, before, warp);
                if ((mine >> lane) & 1u)
                    src_of[b + __popc(mine & ((1u << lane) - 1u))] = (unsigned char)(warp * 32 + lane);
            }
        }
        const int64_t sg = i0 / kCmpSeg;
        int64_t dst = off.blocks > 0 ? (int64_t)(blk_off[sg / kCmpBlockSegs] + __ldg(off.local + sg))
                                     : (int64_t)__ldg(off.global + sg);
        if (SEGU > 1 && u % SEGU != 0) {  // kept in the segment's earlier unit
            const uint32_t w0 = lane < UW ? __ldg(mask + (u - 1) * UW + lane) : 0u;
            dst += __reduce_add_sync(0xffffffffu, (unsigned)__popc(w0));
        }
        __syncthreads();  // src_of, and what plain loads brought
        const int nb = (kept + 31) >> 5;
        int src[UW];
#pragma unroll
        for (int b = 0; b < UW; ++b) src[b] = b * 32 + lane < kept ? src_of[b * 32 + lane] : 0;
        if (out_idx && warp < nb && warp * 32 + lane < kept)
            out_idx[dst + warp * 32 + lane] = (int32_t)(i0 + src_of[warp * 32 + lane]);
        if (!mbar_wait_bounded(&bar, phase)) {
            set_status(status, kEtimeout);
            mbar_wait_bounded(&bar, phase);  // give the copies a second bound before leaving
            return;
        }
        phase ^= 1u;
        for (int r = warp; r < 59; r += kCmpWarps) {
            const unsigned char *t = tile + row_base[r];
            if (CmpRows<DT>::f32(r)) {
                float *o = (r < 3 ? reinterpret_cast<float *>(out_pos) + (int64_t)r * OS
                                  : reinterpret_cast<float *>(out_attr) + (int64_t)(r - 3) * OS) + dst + lane;
#pragma unroll
                for (int b = 0; b < UW; ++b)
                    if (b * 32 + lane < kept) o[b * 32] = *reinterpret_cast<const float *>(t + 4 * src[b]);
            } else {
                constexpr int NF = attr_f32_rows(DT);
                unsigned short *o = reinterpret_cast<unsigned short *>(out_attr + (int64_t)NF * OS * 4) +
                                    (int64_t)(r - 3 - NF) * OS + dst + lane;
#pragma unroll
                for (int b = 0; b < UW; ++b)
                    if (b * 32 + lane < kept) o[b * 32] = *reinterpret_cast<const unsigned short *>(t + 2 * src[b]);
            }
        }
        __syncthreads();  // the tile and src_of are free again
    }
}

template <int DT>
static cudaError_t launch_compact_t(const refine_scene &in, const uint32_t *mask, const CmpOffsets &off, float *out_pos,
                                    void *out_attr, int64_t OS, int32_t *out_idx, int num_sms, int *status, const Chain &s)
{
    const size_t smem = CmpRows<DT>::kBytes;
    static_assert(CmpRows<DT>::kBytes < 40 * 1024, "no opt-in shared memory");
    int64_t g = (in.n + cmp_unit(DT) - 1) / cmp_unit(DT);
    if (g > (int64_t)num_sms * kCmpCtas) g = (int64_t)num_sms * kCmpCtas;
    if (g < 1) g = 1;
    const CmpRows<DT> rows(in.pos, in.attr, in.row_stride, in.n);
    return launch_chained(k_compact<DT>, (int)g, kCmpThreads, smem, s, rows, in.n, mask, off,
                          reinterpret_cast<char *>(out_pos), static_cast<char *>(out_attr), OS, out_idx, status);
}

cudaError_t launch_compact_scatter(const refine_scene &in, const uint32_t *mask, const CmpOffsets &off, float *out_pos,
                                   void *out_attr, int64_t OS, int32_t *out_idx, int num_sms, int *status, const Chain &s)
{
    if (in.dtype == REFINE_BF16)
        return launch_compact_t<REFINE_BF16>(in, mask, off, out_pos, out_attr, OS, out_idx, num_sms, status, s);
    if (in.dtype == REFINE_BF16S)
        return launch_compact_t<REFINE_BF16S>(in, mask, off, out_pos, out_attr, OS, out_idx, num_sms, status, s);
    return launch_compact_t<REFINE_F32>(in, mask, off, out_pos, out_attr, OS, out_idx, num_sms, status, s);
}

}  // namespace refine
