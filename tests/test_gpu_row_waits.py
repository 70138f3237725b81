"""The bounded waits of the kernels that bring rows by bulk copies (the bfloat16
feature pass and the compaction), compiled here with barriers that expect 16
bytes more than come and waits of about a millisecond: the kernels report
REFINE_ETIMEOUT and return, the processing order that the later kernels index
with is a permutation all the same, and the device goes on working.  (The
copies themselves are those of the library and have long landed by then.)"""
import subprocess

import pytest

from paper_2606_09074_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r'''
#include <cstdio>
#include <vector>
#include "common.cuh"
namespace refine {
__device__ __forceinline__ void mbar_expect_more(uint64_t *bar, uint32_t bytes) { mbar_expect_tx(bar, bytes + 16u); }
__device__ __forceinline__ bool mbar_wait_short(uint64_t *bar, uint32_t parity) { return mbar_wait_bounded(bar, parity, 2000000); }
}
#define mbar_expect_tx mbar_expect_more
#define mbar_wait_bounded mbar_wait_short
#include "kernels_prep.cu"
#include "kernels_stream.cu"
using namespace refine;

template <typename T>
static T *device(size_t count)
{
    void *p = nullptr;
    return cudaMalloc(&p, sizeof(T) * count) == cudaSuccess && cudaMemset(p, 0, sizeof(T) * count) == cudaSuccess
               ? static_cast<T *>(p) : nullptr;
}

int main(int argc, char **argv)
{
    int sms = 0, code = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0);
    const int64_t n = 2048 * (int64_t)sms + 20001, S = argc > 1 ? (n + 7) / 8 * 8 : n;  // aligned rows or odd ones
    const int bits = cell_bits_for(n), keys = order_keys(bits);
    float *pos = device<float>(3 * S);
    uint16_t *attr = device<uint16_t>(56 * S);
    refine_camera cam{}, *cams = device<refine_camera>(1);
    for (int k = 0; k < 9; k += 4) cam.R[k] = 1.f;
    cam.fx = cam.fy = cam.cx = cam.cy = cam.zfar = 100.f;
    cam.width = cam.height = 200;
    cam.znear = 0.1f;
    CamRec *rec = device<CamRec>(1);
    OrderGrid *grid = device<OrderGrid>(1);
    PrimRec *recs = device<PrimRec>(n);
    float2 *partials = device<float2>(kFeatSums * 1024);
    SceneConsts *consts = device<SceneConsts>(1);
    SceneStats *stats = device<SceneStats>(1);
    uint2 *cell = device<uint2>(n);
    unsigned *counts = device<unsigned>(keys + 64), *off_local = device<unsigned>(keys), *bsum = device<unsigned>(keys / kScanCells);
    uint32_t *perm = device<uint32_t>(n), *mask = device<uint32_t>((n + 31) / 32);
    int *status = device<int>(1);
    const int blocks = cmp_blocks(n), segs = (int)((n + kCmpSeg - 1) / kCmpSeg);
    unsigned *local = device<unsigned>(segs), *totals = device<unsigned>(blocks);
    CmpState *state = device<CmpState>(1);
    float *out_pos = device<float>(3 * n);
    uint16_t *out_attr = device<uint16_t>(56 * n);
    bool ok = pos && attr && cams && rec && grid && recs && partials && consts && stats && cell && counts && off_local && bsum &&
              perm && mask && status && local && totals && state && out_pos && out_attr &&
              cudaMemcpy(cams, &cam, sizeof cam, cudaMemcpyHostToDevice) == cudaSuccess &&
              cudaMemset(mask, 0xff, 4 * ((n + 31) / 32)) == cudaSuccess &&
              cudaMemset(cell, 0xff, sizeof(uint2) * n) == cudaSuccess;  // what scratch may hold
    if (!ok) return 1;
    PrepLaunch a{};
    a.cams = cams;
    a.V = a.vstride = 1;
    a.cam_out = rec;
    a.cell_bits = bits;
    a.grid = grid;
    a.zero = reinterpret_cast<uint4 *>(counts);
    a.zero4 = (keys + 64) / 4;
    a.status = status;
    const float luma[3] = {0.3f, 0.6f, 0.1f};
    FeatureLaunch f{pos, attr, S, n, 0.05f, luma, recs, partials, grid, bits, cell, counts, status};
    SceneTail tail{};
    tail.partials = partials;
    tail.nblocks = feature_blocks(n);
    tail.n = n;
    tail.p.eta = 0.05f;
    tail.p.e_ln_gem = tail.p.e_col = tail.p.e_opa = 1.0;
    tail.consts = consts;
    tail.stats = stats;
    ok = launch_prepare(pos, attr, REFINE_BF16, S, n, a, sms, nullptr) == cudaSuccess &&
         launch_features(f, REFINE_BF16, sms, nullptr) == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess;
    // the kernels after it index with what it left: looked at before they run
    std::vector<uint2> c(n);
    ok = ok && cudaMemcpy(c.data(), cell, sizeof(uint2) * n, cudaMemcpyDeviceToHost) == cudaSuccess &&
         cudaMemcpy(&code, status, 4, cudaMemcpyDeviceToHost) == cudaSuccess;
    std::vector<unsigned> h(keys);
    ok = ok && cudaMemcpy(h.data(), counts, 4 * keys, cudaMemcpyDeviceToHost) == cudaSuccess;
    int64_t bad = 0, sum = 0;
    for (int k = 0; ok && k < keys; ++k) sum += h[k];
    for (int64_t i = 0; ok && i < n; ++i) bad += c[i].x >= (unsigned)keys || c[i].y >= h[c[i].x < (unsigned)keys ? c[i].x : 0];
    printf("features: status %d, %lld of %lld counted, %lld bad slots\n", code, (long long)sum, (long long)n, (long long)bad);
    if (!ok || code != kEtimeout || sum != n || bad) return 2;
    std::vector<uint32_t> p(n);
    ok = launch_cell_scan(counts, off_local, bsum, counts + keys, bits, nullptr) == cudaSuccess &&
         launch_cell_scatter(cell, n, off_local, bsum, perm, tail, sms, nullptr) == cudaSuccess &&
         cudaMemcpy(p.data(), perm, 4 * n, cudaMemcpyDeviceToHost) == cudaSuccess;
    std::vector<char> seen(n, 0);
    int64_t distinct = 0;
    for (int64_t i = 0; ok && i < n; ++i)
        if (p[i] < n && !seen[p[i]]) seen[p[i]] = 1, ++distinct;
    printf("order: %lld distinct\n", (long long)distinct);
    if (!ok || distinct != n) return 3;
    // the compaction of everything
    std::vector<unsigned> hl(segs), ht(blocks);
    for (int s = 0; s < segs; ++s) hl[s] = (unsigned)(s % kCmpBlockSegs) * kCmpSeg;
    for (int b = 0; b < blocks; ++b) {
        const int64_t left = n - (int64_t)b * kCmpBlockSegs * kCmpSeg;
        ht[b] = (unsigned)(left < kCmpBlockSegs * kCmpSeg ? left : kCmpBlockSegs * kCmpSeg);
    }
    refine_scene in{};
    in.n = n;
    in.dtype = REFINE_BF16;
    in.pos = pos;
    in.attr = attr;
    in.row_stride = S;
    const CmpOffsets off{blocks, local, totals, nullptr, state};
    ok = cudaMemset(status, 0, 4) == cudaSuccess && cudaMemcpy(local, hl.data(), 4 * segs, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(totals, ht.data(), 4 * blocks, cudaMemcpyHostToDevice) == cudaSuccess &&
         launch_compact_scatter(in, mask, off, out_pos, out_attr, n, nullptr, sms, status, nullptr) == cudaSuccess &&
         cudaDeviceSynchronize() == cudaSuccess && cudaMemcpy(&code, status, 4, cudaMemcpyDeviceToHost) == cudaSuccess;
    printf("compaction: status %d\n", code);
    if (!ok || code != kEtimeout) return 4;
    // and the device goes on working
    OrderGrid g;
    ok = launch_prepare(pos, attr, REFINE_BF16, S, n, a, sms, nullptr) == cudaSuccess &&
         cudaMemcpy(&g, grid, sizeof g, cudaMemcpyDeviceToHost) == cudaSuccess && g.qscale[0] == 0.f;
    return ok ? 0 : 5;
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("waits")
    src, exe = d / "waits.cu", d / "waits"
    src.write_text(PROGRAM)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-std=c++17", "--cudart", "shared", "-I", build.INCLUDE, "-I", build.CSRC,
                           str(src), "-o", str(exe)])
    return str(exe)


@pytest.mark.parametrize("rows", ["odd", "aligned"])
def test_row_waits_run_out(program, rows):
    out = subprocess.run([program] + (["aligned"] if rows == "aligned" else []), capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
