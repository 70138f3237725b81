"""The bulk copies that bring a scene's rows into shared memory (RowTile,
rows.cuh) stay within the caller's rows: the address arithmetic itself,
compiled for the host and walked over row strides, column slices, sizes and
units of every storage type.  CPU only."""
import os
import subprocess

from paper_2606_09074_gb300 import build

PROGRAM = r'''
#include <stdio.h>
#include "rows.cuh"
using namespace refine;

static long long bad = 0, copies = 0, narrowed = 0;

// A scene of n columns with rows S elements apart: the caller's memory ends
// with the last row's last column, or, with whole (rows of 8 columns and more
// in whole chunks), with the last chunk that holds some of it.
template <int DT, int U>
static void scene(int64_t n, int64_t S, bool whole_rows = false)
{
    typedef RowTile<DT, U> Rows;
    const char *pos = reinterpret_cast<const char *>(0x100000), *attr = reinterpret_cast<const char *>(0x40000000);
    const int64_t cols = whole_rows ? (n + 7) / 8 * 8 : n;
    const Rows in{pos, attr, S, whole_rows ? Rows::whole_chunks(n) : n};
    const char *pos_end = pos + (2 * S + cols) * 4;
    const int last = (int)attr_f32_rows(DT) == 56 ? 4 : 2;  // bytes of an element of the last row
    const char *attr_end = in.row(58) + cols * last;
    for (int64_t i0 = 0; i0 < n; i0 += U) {
        const int count = (int)(n - i0 < U ? n - i0 : U);
        for (int r = 0; r < 59; ++r) {
            const char *first = in.row(r) + i0 * in.size(r) - in.mis(r);
            const long long bytes = in.span(r, i0, count);
            const char *lo = r < 3 ? pos : attr, *hi = r < 3 ? pos_end : attr_end;
            const bool aligned = ((uintptr_t)first & 15) == 0 && (bytes & 15) == 0;
            const bool inside = bytes == 0 || (first >= lo && first + bytes <= hi);
            const bool fits = bytes <= (in.f32(r) ? Rows::kPitch4 : Rows::kPitch2);
            // every element is brought, or the unit is one whose rest is read by plain loads, at most 7 of a row
            const long long got = (bytes - (long long)in.mis(r)) / in.size(r);
            const bool whole = got >= count || (!whole_rows && Rows::at_end(i0, n) && count - (got > 0 ? got : 0) < 8);
            ++copies;
            narrowed += got < count;
            if (!(aligned && inside && fits && whole) && bad++ < 5)
                printf("DT %d U %d n %lld S %lld unit %lld row %d: aligned %d inside %d fits %d whole %d\n", DT, U,
                       (long long)n, (long long)S, (long long)i0, r, aligned, inside, fits, whole);
        }
    }
}

int main()
{
    const int64_t sizes[] = {1, 2, 3, 7, 8, 9, 15, 16, 17, 120, 127, 128, 129, 248, 249, 255, 256, 257, 263, 264, 265, 511, 513, 770};
    for (int64_t n : sizes)
        for (int64_t S = n; S <= n + 24; ++S) {
            scene<REFINE_F32, 128>(n, S);
            scene<REFINE_F32, 256>(n, S);
            scene<REFINE_BF16, 256>(n, S);
            scene<REFINE_BF16S, 256>(n, S);
            if (S % 8 == 0) {
                scene<REFINE_BF16, 256>(n, S, true);
                scene<REFINE_BF16S, 256>(n, S, true);
            }
        }
    printf("%lld copies, %lld narrowed, %lld bad\n", copies, narrowed, bad);
    return bad != 0;
}
'''


def test_bulk_copies_stay_within_the_rows(tmp_path):
    src, exe = tmp_path / "rows.cu", tmp_path / "rows"
    src.write_text(PROGRAM)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
