"""The plain calls away from ordinary scenes: more views under capture than in
the calls before it; a few primitives far from all others; overflowing pairs; crowded cells."""
import ctypes

import numpy as np
import pytest

import oracle
import test_gpu_parity as parity
from paper_2606_09074_gb300 import synth
from parity_helpers import assert_score_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09074_gb300 import binding as rb
    return torch, rb, torch.device("cuda", 0)


def uploaded(torch, rb, dev, w):
    return torch.from_numpy(w.scene.pos).to(dev), torch.from_numpy(w.scene.attr).to(dev), rb.cameras_to_device(w.cams, dev)


@pytest.mark.parametrize("n", [100_000, 300_000])
def test_capture_with_more_views_than_before(env, n):
    """A captured call may score more views than the calls that sized the
    scratch: what they left holds its scene scratch (512 camera records more
    are 56 KB), and its scores have the bits of an uncaptured call."""
    torch, rb, dev = env
    pos, attr, cams = uploaded(torch, rb, dev, synth.random_scene(seed=n, n=n, v=512, means="core_shell"))
    ref = rb.Context(0)
    want = ref.score(pos, attr, cams)
    torch.cuda.synchronize()
    ctx, stream = rb.Context(0), torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx.score(pos, attr, cams, n_views=64)
        stream.synchronize()
        out = torch.zeros(n, device=dev)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            ctx.score(pos, attr, cams, scores=out)
        for _ in range(2):
            graph.replay()
        stream.synchronize()
        assert torch.equal(out.view(torch.int32), want.view(torch.int32))
        ctx.check()
    ctx.close()
    ref.close()


@pytest.mark.parametrize("n", [900, 200_000])
@pytest.mark.parametrize("rows,value", [("pos", 1e3), ("pos", 1e6), ("pos", -1e9), ("attr", -60.0), ("both", 0.0)])
def test_outliers_leave_the_order_as_it_is(env, n, rows, value):
    """A few primitives far from all others (positions) or far smaller
    (log-scales), among those that the processing order's grid is sampled
    from, leave the other tiles as tight as they were: the pairs decided one
    by one grow by no more than the outliers' own tiles hold.  (Scene 'both'
    mixes three magnitudes of positions with small scales.)"""
    torch, rb, dev = env
    v = 24
    pos, attr, cams = uploaded(torch, rb, dev, synth.random_scene(seed=7, n=n, v=v, means="core_shell"))
    ctx = rb.Context(0)
    _, plain = ctx.score(pos, attr, cams, stats=True)
    # the first and the last four primitives are always among the samples
    far = [0, 1, n - 1]
    for k, i in enumerate(far):
        if rows == "attr":
            attr[0:3, i] = value
        else:
            pos[:, i] = value if rows == "pos" else 10.0 ** (3 + 2 * k)
        if rows == "both":
            attr[0:3, i] = -60.0
    _, got = ctx.score(pos, attr, cams, stats=True)
    ctx.check()
    ctx.close()
    own = len(far) * 64 * v  # each outlier's tile, all pairs
    assert got["mixed_pairs"] <= 1.02 * plain["mixed_pairs"] + own, (got["mixed_pairs"], plain["mixed_pairs"])


def test_far_pair_does_not_depend_on_its_tile(env):
    """A pair so far out that both sides of its footprint test overflow is
    decided the same whether its tile leaves the depth range open or not (a
    second primitive behind the camera opens it)."""
    torch, rb, dev = env
    cam = synth.random_scene(seed=1, n=1, v=1).cams.copy()
    cam["R"], cam["t"] = np.eye(3, dtype=np.float32).reshape(cam["R"].shape), 0.0
    cam["fx"] = cam["fy"] = 500.0
    cam["cx"], cam["cy"], cam["width"], cam["height"] = 320.0, 240.0, 640, 480
    cam["znear"], cam["zfar"] = 0.01, 1e13
    cams = rb.cameras_to_device(cam, dev)
    attr = np.zeros((56, 2), dtype=np.float32)
    attr[0:3], attr[3] = 0.5, 1.0
    pos = np.array([[-4e16, 0.0], [0.0, 0.0], [2e11, -1.0]], dtype=np.float32)
    sums = []
    for n in (1, 2):
        ctx = rb.Context(0)
        vs = torch.zeros(n, device=dev)
        ctx.score(torch.from_numpy(pos[:, :n].copy()).to(dev), torch.from_numpy(attr[:, :n].copy()).to(dev), cams, view_sum=vs)
        ctx.check()
        sums.append(vs[0].item())
        ctx.close()
    assert sums[0] == sums[1] > 0.0


@pytest.mark.parametrize("n,dtype", [(40, "f32"), (5_003, "bf16"), (330_001, "f32"), (330_001, "bf16"), (330_000, "bf16s")])
@pytest.mark.parametrize("kind", ["two", "same", "sorted"])
def test_crowded_cells(env, n, dtype, kind):
    """Centres in a few cells of the processing order's grid (two dense clusters
    far apart, in random and in spatial order, or all in one place): scores
    against the oracle, for the small and the full-grid feature kernels."""
    torch, rb, dev = env
    rng = np.random.default_rng(n)
    w = synth.random_scene(seed=n, n=n, v=3, means="core_shell")
    pos = 0.2 * rng.standard_normal((3, n)) + np.where(rng.random(n) < 0.5, -6.0, 6.0)
    if kind == "same":
        pos[:] = np.array([[0.5], [0.25], [-0.125]])
    elif kind == "sorted":
        pos = pos[:, np.argsort(pos[0])]
    w.scene.pos[:] = pos.astype(np.float32)
    scene = {"f32": w.scene, "bf16": w.scene.to_bf16(), "bf16s": w.scene.to_bf16s()}[dtype]
    pos_d, attr_d, cams = uploaded(torch, rb, dev, w)
    attr_d = {"f32": lambda a: a, "bf16": lambda a: a.to(torch.bfloat16),
              "bf16s": lambda a: rb.MixedRows.from_float(a, device=dev)}[dtype](attr_d)
    ctx, vs = rb.Context(0), torch.empty(n, device=dev)
    got = ctx.score(pos_d, attr_d, cams, view_sum=vs)
    ctx.check()
    ctx.close()
    idx = np.unique(rng.integers(0, n, 2000))
    assert_score_parity(got.cpu().numpy()[idx], vs.cpu().numpy()[idx], oracle.score_subset(scene.params_f64(), idx, w.cams))


@pytest.mark.parametrize("over,dtype", [(3, "f32"), (3, "bf16"), (8, "bf16"), (3, "bf16s")])
def test_chained_large_scenes(env, over, dtype):
    """The plain calls chained, as in test_chained_calls_same_bits, for scenes
    past the small feature kernel's limit."""
    torch, rb, dev = env
    ctx = rb.Context(0)
    n = 2048 * torch.cuda.get_device_properties(dev).multi_processor_count + 8 + over
    parity.test_chained_calls_same_bits(torch, rb, ctx, n, 20, dtype)
    ctx.close()


@pytest.mark.parametrize("n", [196_609, 262_144, 262_145])
def test_unchained_selection_limit(env, n):
    """Sizes about the limit of the one-launch selection in a batch, whose
    kernels are not chained, and the entry point that allocates nothing: the
    masks of the plain call, which takes the passes there."""
    torch, rb, dev = env
    ctx = rb.Context(0)
    pos, attr, cams = uploaded(torch, rb, dev, synth.random_scene(seed=n, n=n, v=2, means="core_shell"))
    b = rb.Batch(ctx, [{"pos": pos, "attr": attr, "cams": cams, "ratio": 0.66}], compact=False)
    for _ in range(2):
        b.run()
    b.results()
    scores = b.outputs[0]["scores"]
    want, thr, nk = ctx.select(scores, 0.66)
    assert torch.equal(b.outputs[0]["mask"], want)
    b.close()
    for s in (scores, torch.floor(4.0 * torch.rand(n, generator=torch.Generator(dev).manual_seed(n), device=dev))):
        want, thr, nk = ctx.select(s, 0.66)
        got = torch.zeros_like(want)
        c_thr, err = ctypes.c_float(), ctypes.create_string_buffer(64)
        assert rb.refine_select_noalloc(s.data_ptr(), n, 0.66, got.data_ptr(), ctypes.byref(c_thr), None, err, 64,
                                        torch.cuda.current_stream().cuda_stream) == rb.REFINE_OK
        assert torch.equal(got, want) and c_thr.value == thr
    ctx.close()
