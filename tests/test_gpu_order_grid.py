"""The processing-order grid that the first kernel of a scene leaves
(launch_prepare), read back by a small program linked against the library."""
import os
import subprocess

import pytest

from paper_2606_09074_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r'''
#include <cmath>
#include <cstdio>
#include <vector>
#include "internal.h"
using namespace refine;

int main()
{
    const int cell_bits = 4, keys = order_keys(cell_bits) + 64;
    OrderGrid *grid;
    CamRec *rec;
    unsigned *counts;
    int *status;
    refine_camera cam{}, *cams;
    for (int k = 0; k < 9; k += 4) cam.R[k] = 1.f;
    cam.fx = cam.fy = cam.cx = cam.cy = 100.f;
    cam.width = cam.height = 200;
    cam.znear = 0.1f;
    cam.zfar = 100.f;
    float *pos, *attr;
    bool ok = cudaMalloc(&grid, sizeof *grid) == cudaSuccess && cudaMalloc(&rec, sizeof *rec) == cudaSuccess &&
              cudaMalloc(&counts, 4 * keys) == cudaSuccess && cudaMalloc(&status, 4) == cudaSuccess &&
              cudaMalloc(&cams, sizeof cam) == cudaSuccess && cudaMalloc(&pos, 3 * 64 * 4) == cudaSuccess &&
              cudaMalloc(&attr, 56 * 64 * 4) == cudaSuccess;
    std::vector<float> h(56 * 64);
    for (size_t i = 0; i < h.size(); ++i) h[i] = 1.f + 0.25f * (float)(i % 64) + 3.f * (float)(i / 64);
    ok = ok && cudaMemcpy(cams, &cam, sizeof cam, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(pos, h.data(), 3 * 64 * 4, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(attr, h.data(), 56 * 64 * 4, cudaMemcpyHostToDevice) == cudaSuccess;
    for (int n = 1; n <= 5 && ok; ++n) {
        PrepLaunch a{};
        a.cams = cams;
        a.V = a.vstride = 1;
        a.cam_out = rec;
        a.cell_bits = cell_bits;
        a.grid = grid;
        a.zero = reinterpret_cast<uint4 *>(counts);
        a.zero4 = keys / 4;
        a.status = status;
        OrderGrid g;
        ok = cudaMemset(grid, 0xff, sizeof *grid) == cudaSuccess;  // NaN
        ok = ok && launch_prepare(pos, attr, REFINE_F32, 64, n, a, 2, nullptr) == cudaSuccess &&
             cudaMemcpy(&g, grid, sizeof g, cudaMemcpyDeviceToHost) == cudaSuccess;
        printf("%d", n);
        for (int k = 0; k < 3; ++k) printf(" %.9g", g.lo[k]);
        for (int k = 0; k < 3; ++k) printf(" %.9g", g.qscale[k]);
        printf(" %.9g\n", g.big_ls);
    }
    return ok ? 0 : 1;
}
'''


@pytest.fixture(scope="module")
def grids(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = build.build_library()
    d = tmp_path_factory.mktemp("grid")
    src, exe = d / "grid.cu", d / "grid"
    src.write_text(PROGRAM)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-std=c++17", "--cudart", "shared", "-I", build.INCLUDE, "-I", build.CSRC,
                           str(src), lib, "-Xlinker", "-rpath," + os.path.dirname(lib), "-o", str(exe)])
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
    return {int(r.split()[0]): [float(x) for x in r.split()[1:]] for r in out.stdout.strip().split("\n")}


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
def test_grid_of_the_smallest_scenes(grids, n):
    """The box is mean - 3 sd and 16 cells over 6 sd on every axis, and the
    large primitives begin above mean + 1.28 sd of ln s_max (the values are
    1 + i / 4 + 3 row: exact in float32, so a rounding or two apart)."""
    i = [0.25 * k for k in range(n)]
    mean = sum(i) / n
    sd = (sum(x * x for x in i) / n - mean * mean) ** 0.5
    lo, qs, big = grids[n][:3], grids[n][3:6], grids[n][6]
    for k in range(3):
        assert lo[k] == pytest.approx(1.0 + 3.0 * k + mean - 3.0 * sd, rel=1e-5, abs=1e-5)
        assert qs[k] == pytest.approx(16.0 / (6.0 * sd) if sd > 0 else 0.0, rel=1e-5)
    # rows 0-2 of attr: the largest log-scale is row 2's
    assert big == pytest.approx(7.0 + mean + 1.28 * sd, rel=1e-5)
