"""Row layouts of scenes large enough for the feature kernels of a full grid
(above 2,048 primitives per SM): strides of every alignment, padded rows and
column slices of a larger block give the bits of rows that start on 16 bytes,
and those agree with the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2606_09074_gb300 import synth
from parity_helpers import assert_score_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09074_gb300 import binding as rb
    ctx = rb.Context(0)
    yield torch, rb, ctx
    ctx.close()


def laid_out(torch, rb, pos, attr, dtype, stride, first):
    """The scene's rows `stride` elements apart, from column `first` of their block."""
    n, dev = pos.shape[1], pos.device
    p = torch.full((3, stride), 7.0, device=dev)
    p[:, first: first + n] = pos
    if dtype == "bf16s":
        a = rb.MixedRows.empty(n, stride=stride, device=dev)
        a.f32_rows()[:, :n] = attr[:3]
        a.bf16_rows()[:, :n] = attr[3:].to(torch.bfloat16)
        return p[:, :n], a
    a = torch.full((56, stride), 7.0, device=dev, dtype=torch.bfloat16 if dtype == "bf16" else torch.float32)
    a[:, first: first + n] = attr.to(a.dtype)
    return p[:, first: first + n], a[:, first: first + n]


@pytest.mark.parametrize("dtype", ["f32", "bf16", "bf16s"])
@pytest.mark.parametrize("over", [-1, 1, 6, 8])
def test_large_row_layouts(env, dtype, over):
    torch, rb, ctx = env
    dev = torch.device("cuda", 0)
    n = 2048 * torch.cuda.get_device_properties(dev).multi_processor_count + over  # the small form ends at over = 0
    w = synth.random_scene(seed=5 + over, n=n, v=4, means="core_shell")
    pos, attr = torch.from_numpy(w.scene.pos).to(dev), torch.from_numpy(w.scene.attr).to(dev)
    cams = rb.cameras_to_device(w.cams, dev)
    n8 = (n + 7) // 8 * 8
    p0, a0 = laid_out(torch, rb, pos, attr, dtype, n8 + 8, 0)
    vs = torch.empty(n, dtype=torch.float32, device=dev)
    want = ctx.score(p0, a0, cams, view_sum=vs)
    mask, _, nk = ctx.select(want, 0.4)
    kept = ctx.compact(p0, a0, mask, nk)
    scene = {"f32": w.scene, "bf16": w.scene.to_bf16(), "bf16s": w.scene.to_bf16s()}[dtype]
    idx = np.unique(np.concatenate([np.arange(300), np.random.default_rng(over + 9).integers(0, n, 3000), np.arange(n - 300, n)]))
    ref = oracle.score_subset(scene.params_f64(), idx, w.cams)
    assert_score_parity(want.cpu().numpy()[idx], vs.cpu().numpy()[idx], ref)
    # (stride, first column); a slice to the end of its block when stride - first = n
    layouts = [(n, 0), (n + 1, 0), (n + 3, 0), (n8, 0)] + ([] if dtype == "bf16s" else [(n + 8, 8), (n + 16, 16), (n + 13, 8)])
    for stride, first in layouts:
        p, a = laid_out(torch, rb, pos, attr, dtype, stride, first)
        got = ctx.score(p, a, cams)
        assert torch.equal(got.view(torch.int32), want.view(torch.int32)), (stride - n, first)
        op, oa, oi = ctx.compact(p, a, mask, nk)
        assert torch.equal(op, kept[0]) and torch.equal(oa.float(), kept[1].float()) and torch.equal(oi, kept[2]), (stride - n, first)
    ctx.check()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "bf16s"])
@pytest.mark.parametrize("n,pad", [(1, 0), (255, 1), (257, 0), (12_345, 3), (200_001, 0)])
def test_compact_units_of_every_count(env, dtype, n, pad):
    """Units of 256 primitives that keep 0 to 12, 31 to 34 or all of theirs
    (those of at most 8 are read element by element, those of at most 32 take
    one store a row), the kept ones at random places, the unit's first and last
    among them: equal to indexing the rows."""
    torch, rb, ctx = env
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(n + pad)
    keep = np.zeros(n, dtype=bool)
    counts = list(range(13)) + [31, 32, 33, 34, 256]
    for u in range(0, n, 256):
        size = min(256, n - u)
        k = min(size, counts[(u // 256) % len(counts)])
        at = rng.permutation(size)[:k]
        if k >= 2:
            at = np.unique(np.concatenate([at[2:], [0, size - 1]]))
        keep[u + at] = True
    keep[n - 1] = True
    words = np.packbits(np.pad(keep, (0, -n % 32)), bitorder="little").view(np.int32)
    want = torch.from_numpy(np.nonzero(keep)[0]).to(dev)
    g = torch.Generator(device=dev).manual_seed(n)
    pos = torch.randn((3, n), generator=g, device=dev)
    attr = torch.randn((56, n), generator=g, device=dev)
    p, a = laid_out(torch, rb, pos, attr, dtype, n + pad, 0)
    rows = a.float()[:, :n]
    for with_idx in (True, False):
        op, oa, oi, cnt = ctx.compact(p, a if dtype != "bf16s" else a[:, :n], torch.from_numpy(words).to(dev), want.numel(),
                                      out_row_stride=want.numel() + pad, kept_idx=with_idx, return_count=True)
        assert cnt == want.numel()
        assert oi is None if not with_idx else torch.equal(oi, want.to(torch.int32))
        assert torch.equal(op, p[:, want]) and torch.equal(oa.float(), rows[:, want])
