// Compaction, pass 2: the scatter of every row of the kept primitives.
//
// One CTA of 8 warps takes a unit of 256 consecutive primitives at a time.
// The unit's span of each of the 59 rows, 512 or 1,024 contiguous bytes, is
// brought into shared memory by one bulk copy (cp.async.bulk) per row,
// completing on an mbarrier (RowTile); meanwhile the ranks of the kept
// primitives are inverted (output d comes from primitive src[d]).  Then each
// warp takes every eighth row: 32 outputs are one shared-memory load and one
// contiguous store.  A unit is 31-34 KB with bfloat16 rows and 64 KB with
// float32 ones, so 5 or 3 CTAs fit an SM, and while some wait for their unit
// others store theirs: 155-190 KB an SM in flight without holding a register.
// Of a unit with at most kCmpFew kept primitives only their own sectors are
// read, by plain loads.
//
// Measured (count and scatter, cold L2, kept at random; us at ratio 0 / 0.5 /
// 0.9 / 0.98 / 0.995):
//   3.5M float32   272 / 201 / 149 /  92 /  55   (units of 128, all copied whole:
//                  282 / 219 / 174 / 166 / 104; a warp for 256 primitives, rows
//                  through registers: 272 / 222 / 187 / 178 / 173)
//   3.5M bfloat16  156 / 113 /  90 /  74 /  45   (all units copied whole, 6 CTAs
//                  of 40 registers: 158 / 118 / 102 / 100 /  86; a warp for 32
//                  primitives: 210 / 182 / 159 / 118 /  69)
//   1M float32      84 /  66 /  53 /  35 /  23   (86 / 68 / 57 / 55 / 39 and
//                   92 /  82 /  69 /  51 /  36)
// Units of at most 4 kept primitives instead of 8: 3.5M float32 133 us at 0.98;
// at most 16: 164 us at 0.9.
#include <type_traits>

#include "internal.h"
#include "rows.cuh"

namespace refine {

constexpr int kCmpWarps = 8;
constexpr int kCmpThreads = 32 * kCmpWarps;
constexpr int kCmpUnit = kCmpSeg;  // primitives per unit
constexpr int kCmpFew = 8;
// Per SM: what fits its shared memory with float32 rows, registers (48 a
// thread) with bfloat16 ones.
__host__ __device__ constexpr int cmp_ctas(int dtype) { return dtype == REFINE_F32 ? 3 : 5; }

template <int DT>
using CmpRows = RowTile<DT, kCmpUnit>;

// The rows of a unit's `kept` (at most kCmpFew) primitives by loads of their
// own: every group of kCmpFew threads takes a row.  word: the unit's mask, a
// word per lane from lane `at` on.
template <int DT>
__device__ __forceinline__ void copy_few(const CmpRows<DT> &in, int64_t i0, uint32_t word, int at, int kept, int64_t dst,
                                         char *out_pos, char *out_attr, int64_t OS, int32_t *out_idx)
{
    constexpr int kRows = kCmpThreads / kCmpFew, kTurns = (59 + kRows - 1) / kRows, NF = attr_f32_rows(DT);
    const int d = threadIdx.x % kCmpFew;
    // the d-th kept primitive: its word, and its rank there
    int left = d, rank = 0;
    int64_t i = i0;
    uint32_t mine = 0u;
#pragma unroll
    for (int w = 0; w < kCmpUnit / 32; ++w) {
        const uint32_t m = __shfl_sync(0xffffffffu, word, at + w);
        const int c = __popc(m);
        if (left >= 0 && left < c) {
            mine = m;
            rank = left;
            i = i0 + w * 32;
        }
        left -= c;
    }
    if (d >= kept) return;
    for (int k = 0; k < rank; ++k) mine &= mine - 1u;
    i += __ffs(mine) - 1;
    dst += d;
    if (out_idx && threadIdx.x < kCmpFew) out_idx[dst] = (int32_t)i;
    uint32_t v[kTurns];
#pragma unroll
    for (int k = 0; k < kTurns; ++k) {
        const int r = threadIdx.x / kCmpFew + k * kRows;
        if (r >= 59) continue;
        v[k] = in.f32(r) ? __ldg(reinterpret_cast<const uint32_t *>(in.row(r)) + i)
                         : __ldg(reinterpret_cast<const unsigned short *>(in.row(r)) + i);
    }
#pragma unroll
    for (int k = 0; k < kTurns; ++k) {
        const int r = threadIdx.x / kCmpFew + k * kRows;
        if (r >= 59) continue;
        if (in.f32(r))
            *((r < 3 ? reinterpret_cast<uint32_t *>(out_pos) + r * OS
                     : reinterpret_cast<uint32_t *>(out_attr) + (r - 3) * OS) + dst) = v[k];
        else
            reinterpret_cast<unsigned short *>(out_attr + NF * OS * 4)[(r - 3 - NF) * OS + dst] = (unsigned short)v[k];
    }
}

template <int DT>
__global__ void __launch_bounds__(kCmpThreads, cmp_ctas(DT)) k_compact(CmpRows<DT> in, int64_t n, const uint32_t *__restrict__ mask,
                                                         CmpOffsets off, char *__restrict__ out_pos,
                                                         char *__restrict__ out_attr, int64_t OS,
                                                         int32_t *__restrict__ out_idx, int *status)
{
    constexpr int UNIT = kCmpUnit, UW = UNIT / 32;
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
    auto start_of = [&](int64_t u) {  // where the unit's first kept primitive goes
        return off.blocks > 0 ? (int64_t)(blk_off[u / kCmpBlockSegs] + __ldg(off.local + u)) : (int64_t)__ldg(off.global + u);
    };
    bool few = false;
    uint32_t next_word = load_word(blockIdx.x);
    for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
        const uint32_t word = next_word;
        next_word = load_word(u + gridDim.x);
        const int kept = __reduce_add_sync(0xffffffffu, (unsigned)__popc(word));
        if (kept <= kCmpFew) {  // the same in every thread
            few |= kept > 0;
            continue;
        }
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
        const int64_t dst = start_of(u);
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
        // The rows of the tile to their places, 32 outputs at a time.  (Left
        // to the compiler, whether the row loop was unrolled hung on code far
        // from it: 158 or 184 us, 3.5M bfloat16 at ratio 0.)
        auto put = [&](auto words, auto *out, int r) {
            using E = std::remove_pointer_t<decltype(out)>;
            const unsigned char *t = tile + row_base[r];
#pragma unroll
            for (int b = 0; b < decltype(words)::value; ++b)
                if (b * 32 + lane < kept) out[b * 32] = *reinterpret_cast<const E *>(t + sizeof(E) * src[b]);
        };
        constexpr int NF = CmpRows<DT>::kF32;
        auto put_rows = [&](auto words) {
#pragma unroll 2
            for (int r = warp; r < NF; r += kCmpWarps)
                put(words, (r < 3 ? reinterpret_cast<float *>(out_pos) + r * OS
                                  : reinterpret_cast<float *>(out_attr) + (r - 3) * OS) + dst + lane, r);
            unsigned short *out2 = reinterpret_cast<unsigned short *>(out_attr + (NF - 3) * OS * 4) + dst + lane;
#pragma unroll 7
            for (int r = NF + warp; r < 59; r += kCmpWarps) put(words, out2 + (r - NF) * OS, r);
        };
        if (kept <= 32)
            put_rows(std::integral_constant<int, 1>());
        else
            put_rows(std::integral_constant<int, UW>());
        __syncthreads();  // the tile and src_of are free again
    }
    if (!few) return;

    // The units with few kept primitives, in a loop of their own: within the
    // other it took registers from it.  No barrier: the warps go through them
    // on their own, the words of four units at a time (lane l: word l % UW of the
    // l / UW-th), so that a unit with nothing to copy costs a quarter of a load's
    // latency: 30M bfloat16 at ratio 0.999 259 us with one unit at a time.  (In
    // the main loop that cost the load of the next word ahead: 30M at 0.5 1,010
    // against 1,168 us.)
    const int64_t step = gridDim.x;
    for (int64_t u0 = blockIdx.x; u0 < units; u0 += 32 / UW * step) {
        const int64_t un = u0 + lane / UW * step, w = un * UW + lane % UW;
        uint32_t word = 0u;
        if (un < units && w < words) {
            word = __ldg(mask + w);
            const int64_t valid = n - w * 32;
            if (valid < 32) word &= (1u << valid) - 1u;
        }
        int kept = __popc(word);
#pragma unroll
        for (int o = 1; o < UW; o <<= 1) kept += __shfl_xor_sync(0xffffffffu, kept, o);
        for (unsigned todo = __ballot_sync(0xffffffffu, lane % UW == 0 && kept > 0 && kept <= kCmpFew); todo; todo &= todo - 1u) {
            const int at = __ffs(todo) - 1;
            const int64_t u = u0 + at / UW * step;
            copy_few<DT>(in, u * UNIT, word, at, __shfl_sync(0xffffffffu, kept, at), start_of(u), out_pos, out_attr, OS,
                         out_idx);
        }
    }
}

template <int DT>
static cudaError_t launch_compact_t(const refine_scene &in, const uint32_t *mask, const CmpOffsets &off, float *out_pos,
                                    void *out_attr, int64_t OS, int32_t *out_idx, int num_sms, int *status, const Chain &s)
{
    const size_t smem = CmpRows<DT>::kBytes;
    if (smem + 4 * 1024 > 48 * 1024) {  // static part included; one constant for every launch
        const cudaError_t e = cudaFuncSetAttribute(k_compact<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int64_t g = (in.n + kCmpUnit - 1) / kCmpUnit;
    if (g > (int64_t)num_sms * cmp_ctas(DT)) g = (int64_t)num_sms * cmp_ctas(DT);
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
