// A unit of consecutive primitives in shared memory: its span of each of the
// 59 rows, brought by one bulk copy (cp.async.bulk) a row.  A bulk copy starts
// on 16 bytes: the row's span is widened to 16-byte boundaries (row strides may
// be odd) and its place in shared memory is taken from its misalignment.  At
// a scene's end the widened span of the last row of a block could pass the
// row's last element, where the caller's memory may end (a scene may be a
// column slice that reaches the end of its block; of the last few rows, when
// the stride is below 8): it is narrowed instead, and its last few elements are
// read by plain loads.
#pragma once

#include "common.cuh"

namespace refine {

// The rows of a scene in units of U primitives: rows 0-2 the means, then the
// attribute rows; the first kF32 rows are float32, the others bfloat16.
template <int DT, int U>
struct RowTile {
    static constexpr int kF32 = 3 + attr_f32_rows(DT);
    // a row's span and 16 bytes for its misalignment
    static constexpr int kPitch4 = 4 * U + 16, kPitch2 = 2 * U + 16;
    static constexpr int kBytes = kF32 * kPitch4 + (59 - kF32) * kPitch2;

    const char *pos, *attr;
    int64_t S;
    const char *pos_end, *attr_end;  // past the last element of the last row of each block

    // The first n columns of rows S elements apart.
    __host__ RowTile(const void *p, const void *a, int64_t stride, int64_t n)
        : pos(static_cast<const char *>(p)), attr(static_cast<const char *>(a)), S(stride), pos_end(row(2) + n * 4),
          attr_end(row(58) + n * size(58))
    {
    }

    __host__ __device__ static constexpr bool f32(int r) { return r < kF32; }
    __host__ __device__ static constexpr int size(int r) { return r < kF32 ? 4 : 2; }
    __host__ __device__ static constexpr int place(int r)  // byte offset in the tile
    {
        return r < kF32 ? r * kPitch4 : kF32 * kPitch4 + (r - kF32) * kPitch2;
    }
    __host__ __device__ __forceinline__ const char *row(int r) const
    {
        constexpr int NF = attr_f32_rows(DT);
        if (r < 3) return pos + (int64_t)r * S * 4;
        if (r - 3 < NF) return attr + (int64_t)(r - 3) * S * 4;
        return attr + (int64_t)NF * S * 4 + (int64_t)(r - 3 - NF) * S * 2;
    }
    // Bytes of row r past a 16-byte boundary (the same at every unit's start).
    __host__ __device__ __forceinline__ uint32_t mis(int r) const
    {
        return (uint32_t)(reinterpret_cast<uintptr_t>(row(r)) & 15u);
    }
    // Bytes of the bulk copy of `count` elements of row r from element i0: up
    // to the next 16-byte boundary, or down to the last when that lies past
    // the end of the row's block.
    __host__ __device__ __forceinline__ uint32_t span(int r, int64_t i0, int count) const
    {
        const uint32_t m = mis(r), b = m + (uint32_t)(count * size(r)), up = (b + 15u) & ~15u;
        return row(r) + i0 * size(r) - m + up > (r < 3 ? pos_end : attr_end) ? b & ~15u : up;
    }
    // With a stride that is a multiple of 8, for n: so many elements of every
    // row are in whole 16-byte chunks of the block that the rows are from, so
    // copies up to them need no narrowing (a slice of the block starts on 16
    // bytes, that is on a multiple of 8 columns when it has 2-byte rows).
    __host__ __device__ __forceinline__ static int64_t whole_chunks(int64_t n) { return (n + 7) & ~int64_t(7); }
    // Whether some copy of the unit at i0 may be narrowed.
    __host__ __device__ __forceinline__ static bool at_end(int64_t i0, int64_t n) { return i0 + U + 8 > n; }

    // Issues the copies of the unit at i0 (a multiple of U), completing on
    // `bar`; called by every warp of a CTA of WARPS warps, after a barrier that
    // ends all earlier accesses to the tile.  The lanes of a warp issue bulk
    // copies one after the other (some 40 cycles each), so the rows are dealt
    // to all warps; a copy may end before warp 0 has told the barrier how many
    // bytes to expect, as the phase also waits for that arrival.
    template <int WARPS>
    __device__ __forceinline__ void stage(unsigned char *tile, int64_t i0, int count, uint64_t *bar) const
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        fence_proxy_async_shared();  // the tile was accessed by plain loads and stores
        const int r = warp + WARPS * lane;
        const uint32_t mine = r < 59 ? span(r, i0, count) : 0u;
        if (mine > 0u) bulk_g2s(tile + place(r), row(r) + i0 * size(r) - mis(r), mine, bar);
        if (warp == 0) {
            uint32_t bytes = span(lane, i0, count) + (lane + 32 < 59 ? span(lane + 32, i0, count) : 0u);
            bytes = __reduce_add_sync(0xffffffffu, bytes);
            if (lane == 0) mbar_expect_tx(bar, bytes);
        }
    }
    // What narrowed copies leave (fewer than 8 elements a row), by every warp;
    // the caller puts a barrier before the tile is read.
    template <int WARPS>
    __device__ __forceinline__ void rest(unsigned char *tile, int64_t i0, int count) const
    {
        const int lane = threadIdx.x & 31;
        for (int r = threadIdx.x >> 5; r < 59; r += WARPS) {
            const int j = max(0, (int)span(r, i0, count) - (int)mis(r)) / size(r) + lane;
            if (j >= count) continue;
            if (f32(r))
                *reinterpret_cast<float *>(tile + place(r) + mis(r) + 4 * j) =
                    __ldg(reinterpret_cast<const float *>(row(r)) + i0 + j);
            else
                *reinterpret_cast<unsigned short *>(tile + place(r) + mis(r) + 2 * j) =
                    __ldg(reinterpret_cast<const unsigned short *>(row(r)) + i0 + j);
        }
    }
};

}  // namespace refine
