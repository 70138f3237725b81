"""GPU parity: the CUDA path through the C ABI against the FP64 oracle.

Tolerances: float32 scores within 1e-5 relative of the oracle for every
primitive whose visibility decisions are all outside the oracle's float32
band; primitives with a borderline pair must equal the oracle's sum with
some choice of those pairs.  Selection and compaction on identical scores
are bit-exact.  Masks from the oracle's own scores agree except for
primitives within 1e-5 of the threshold or with a borderline pair."""
import ctypes
import math
import os

import numpy as np
import pytest

import oracle
from paper_2606_09074_gb300 import synth
from parity_helpers import RTOL, assert_score_parity, check_mask_vs_oracle_scores, unpack

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


@pytest.fixture(scope="module")
def rb(torch):
    from paper_2606_09074_gb300 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(rb):
    c = rb.Context(0)
    yield c
    c.close()


def upload(torch, rb, scene, cams):
    dev = torch.device("cuda", 0)
    pos = torch.from_numpy(np.ascontiguousarray(scene.pos)).to(dev)
    if scene.dtype == "bf16":
        attr = torch.from_numpy(np.ascontiguousarray(scene.attr).view(np.int16)).to(dev).view(torch.bfloat16)
    elif scene.dtype == "bf16s":
        attr = rb.MixedRows.from_float(scene.attr, device=dev)
    else:
        attr = torch.from_numpy(np.ascontiguousarray(scene.attr)).to(dev)
    return pos, attr, rb.cameras_to_device(cams, dev)


def gpu_score(torch, rb, ctx, scene, cams, params=None):
    pos, attr, cd = upload(torch, rb, scene, cams)
    vs = torch.empty(max(scene.n, 1), dtype=torch.float32, device=pos.device)
    sc, st = ctx.score(pos, attr, cd, params=params, view_sum=vs, stats=True)
    ctx.check()
    return sc.cpu().numpy(), vs[: scene.n].cpu().numpy(), st, (pos, attr)


def oracle_params_from(p, rb):
    if p is None:
        return oracle.params()
    return oracle.params(eta=float(np.float32(p.eta)), e_ln_gem=p.e_ln_gem, e_col=p.e_col, e_opa=p.e_opa,
                         luma=[float(np.float32(x)) for x in p.luma], flags=p.flags)


def check_select_exact(torch, ctx, s_gpu, ratio):
    t = torch.from_numpy(s_gpu.astype(np.float32)).cuda()
    mask, thr, nk = ctx.select(t, ratio)
    m_ref, thr_ref, nk_ref = oracle.select(s_gpu.astype(np.float64), ratio)
    n = s_gpu.shape[0]
    assert nk == nk_ref == n - math.floor(ratio * n)
    got = mask.cpu().numpy().view(np.uint32)[: (n + 31) // 32]
    assert np.array_equal(got, m_ref), "keep mask differs from the oracle on identical scores"
    assert thr == np.float32(thr_ref)  # also covers -inf (nothing pruned) and +inf
    return mask, got, nk


def check_compact_exact(torch, ctx, scene, pos, attr, mask, nk):
    op, oa, idx, cnt = ctx.compact(pos, attr, mask, nk, return_count=True)
    assert cnt == nk
    m = mask.cpu().numpy().view(np.uint32)[: (scene.n + 31) // 32]
    kp, ki = oracle.compact(np.ascontiguousarray(scene.pos), m)
    ka, _ = oracle.compact(np.ascontiguousarray(scene.attr), m)
    assert np.array_equal(idx.cpu().numpy(), ki)
    assert np.array_equal(op.cpu().numpy(), kp)
    got_attr = oa.cpu()
    if scene.dtype == "bf16":
        got_attr = got_attr.view(torch.int16).numpy().view(np.uint16)
    elif scene.dtype == "bf16s":
        got_attr = got_attr.float().numpy()  # widened exactly, rows 3..55 from bfloat16
    else:
        got_attr = got_attr.numpy()
    assert np.array_equal(got_attr, ka)


# ----------------------------------------------------------------- tests

def test_small_scene_full_parity(torch, rb, ctx):
    """N=10k, V=16 ring at 640x480: every score, the scene statistics, the
    selection and the compaction."""
    w = synth.config0()
    s, S, st, (pos, attr) = gpu_score(torch, rb, ctx, w.scene, w.cams)
    ref = oracle.score(w.scene.params_f64(), w.cams)
    clean = assert_score_parity(s, S, ref)
    assert clean.mean() > 0.99
    for k in ("F_col", "F_opa", "F_gem"):
        assert st[k] == pytest.approx(ref["stats"][k], rel=1e-6)
    np.testing.assert_allclose(st["lambda"], ref["stats"]["lambda"], rtol=1e-6)
    np.testing.assert_allclose(st["mean_m"], ref["stats"]["mean_m"], rtol=1e-6)
    mask, words, nk = check_select_exact(torch, ctx, s, 0.5)
    agree = check_mask_vs_oracle_scores(words, ref, 0.5, w.scene.n)
    assert agree > 0.999
    check_compact_exact(torch, ctx, w.scene, pos, attr, mask, nk)


@pytest.mark.parametrize("n,v", [(1, 1), (2, 3), (31, 16), (33, 17), (257, 5), (1023, 33), (4097, 2), (6001, 48)])
def test_ragged_sizes(torch, rb, ctx, n, v):
    w = synth.random_scene(seed=n * 31 + v, n=n, v=v)
    s, S, _, (pos, attr) = gpu_score(torch, rb, ctx, w.scene, w.cams)
    ref = oracle.score(w.scene.params_f64(), w.cams)
    assert_score_parity(s, S, ref)
    for ratio in (0.0, 0.3, 0.5, 0.9):
        mask, _, nk = check_select_exact(torch, ctx, s, ratio)
        check_compact_exact(torch, ctx, w.scene, pos, attr, mask, nk)


def test_bf16_storage_parity(torch, rb, ctx):
    """BF16 rows 3-58: the oracle sees the same bf16-rounded numbers."""
    w = synth.config0(seed=4)
    sc = w.scene.to_bf16()
    s, S, _, (pos, attr) = gpu_score(torch, rb, ctx, sc, w.cams)
    ref = oracle.score(sc.params_f64(), w.cams)
    assert_score_parity(s, S, ref)
    mask, _, nk = check_select_exact(torch, ctx, s, 0.66)
    check_compact_exact(torch, ctx, sc, pos, attr, mask, nk)


def test_bf16s_storage_parity(torch, rb, ctx):
    """Log-scale rows float32, rows 6-58 bfloat16 (REFINE_BF16S): the oracle
    sees the same numbers; selection and compaction are exact, the mixed
    rows included; and the log-scales reach the kernels unrounded (the
    scores differ from the all-BF16 form's wherever a log-scale is not a
    bfloat16 value)."""
    w = synth.config0(seed=4)
    sc = w.scene.to_bf16s()
    assert np.array_equal(sc.attr[:3], w.scene.attr[:3])
    s, S, _, (pos, attr) = gpu_score(torch, rb, ctx, sc, w.cams)
    ref = oracle.score(sc.params_f64(), w.cams)
    assert_score_parity(s, S, ref)
    mask, _, nk = check_select_exact(torch, ctx, s, 0.66)
    check_compact_exact(torch, ctx, sc, pos, attr, mask, nk)
    sb = gpu_score(torch, rb, ctx, w.scene.to_bf16(), w.cams)[0]
    assert not np.array_equal(s, sb)


@pytest.mark.parametrize("n,v", [(1, 3), (1000, 7), (33_333, 40)])
def test_bf16s_ragged_and_host_path(torch, rb, ctx, n, v):
    """Ragged sizes in the mixed layout, and the whole pass from host rows
    (refine_prune_host) equal to the device path."""
    w = synth.random_scene(seed=n + v, n=n, v=v, means="core_shell")
    sc = w.scene.to_bf16s()
    s, S, _, (pos, attr) = gpu_score(torch, rb, ctx, sc, w.cams)
    assert_score_parity(s, S, oracle.score(sc.params_f64(), w.cams))
    mask, thr, nk = ctx.select(torch.from_numpy(s).cuda(), 0.5)
    op, oa, idx = ctx.compact(pos, attr, mask, nk)
    r = ctx.prune_host(torch.from_numpy(sc.pos).pin_memory(), rb.MixedRows.from_float(sc.attr, pin_memory=True),
                       w.cams, 0.5, want_scores=True)
    assert r["n_keep"] == nk and r["threshold"] == thr
    assert np.array_equal(r["scores"].numpy().view(np.uint32), s.view(np.uint32))
    assert np.array_equal(r["idx"].numpy(), idx.cpu().numpy())
    assert np.array_equal(r["out_pos"].numpy(), op.cpu().numpy())
    assert torch.equal(r["out_attr"].float(), oa.float().cpu())


def test_many_views_multipass(torch, rb, ctx):
    """More views than one launch stages (1024): the view set is split."""
    w = synth.random_scene(seed=8, n=700, v=1100)
    s, S, _, _ = gpu_score(torch, rb, ctx, w.scene, w.cams)
    ref = oracle.score(w.scene.params_f64(), w.cams)
    assert_score_parity(s, S, ref)


def test_ablation_flags(torch, rb, ctx):
    """Table 3 modes and the Eq. 14 Jacobian energy (FULL_JACOBIAN, for which
    NO_PROJ takes precedence) against the oracle."""
    w = synth.config0(seed=5, n=3000)
    # The Jacobian energy grows as 1/z^4: float32's cancellation error in
    # z = R2 mu + t2 (relative 2^-24 (|R2||mu| + |t2|) / z) is amplified four
    # times, so its cameras keep z >= 1 (znear = 1), where that bound stays
    # under 1e-6 for these scenes.
    far_cams = w.cams.copy()
    far_cams["znear"] = 1.0
    for flags in (rb.FLAG_NORM_ATTR | rb.FLAG_NO_VIS, rb.FLAG_NORM_ATTR | rb.FLAG_NO_PROJ,
                  rb.FLAG_NORM_ATTR | rb.FLAG_EQUAL_LAMBDA, 0, rb.FLAG_NORM_ATTR | rb.FLAG_FULL_JACOBIAN,
                  rb.FLAG_NORM_ATTR | rb.FLAG_FULL_JACOBIAN | rb.FLAG_NO_PROJ):
        p = rb.default_params(flags=flags)
        cams = far_cams if flags & rb.FLAG_FULL_JACOBIAN else w.cams
        s, S, _, _ = gpu_score(torch, rb, ctx, w.scene, cams, params=p)
        ref = oracle.score(w.scene.params_f64(), cams, oracle_params_from(p, rb))
        assert_score_parity(s, S, ref)


def test_degenerate_scales(torch, rb, ctx):
    """Scales that underflow float32 (flat discs and needles)."""
    w = synth.random_scene(seed=9, n=300, v=12)
    sc = w.scene
    sc.attr[0, 0:40] = -200.0               # disc: one zero scale
    sc.attr[0:2, 40:80] = -200.0            # needle: two zero scales
    sc.attr[0:3, 80:90] = -200.0            # point: three zero scales
    s, S, _, _ = gpu_score(torch, rb, ctx, sc, w.cams)
    ref = oracle.score(sc.params_f64(), w.cams)
    assert_score_parity(s, S, ref)


def test_empty_scene(torch, rb, ctx):
    w = synth.random_scene(seed=1, n=1, v=2)
    dev = torch.device("cuda", 0)
    pos = torch.zeros((3, 0), device=dev)
    attr = torch.zeros((56, 0), device=dev)
    cams = rb.cameras_to_device(w.cams, dev)
    s = ctx.score(pos, attr, cams)
    assert s.numel() == 0
    mask, thr, nk = ctx.select(s, 0.5)
    assert nk == 0 and math.isinf(thr)
    ctx.check()


def test_select_edge_inputs(torch, rb, ctx):
    rng = np.random.default_rng(3)
    cases = {
        "equal": np.full(5000, 0.25, dtype=np.float32),
        "zeros_heavy": np.where(rng.random(70001) < 0.7, 0.0, rng.random(70001)).astype(np.float32),
        "signed_zero": np.where(rng.random(9000) < 0.5, -0.0, 0.0).astype(np.float32),
        "negative": rng.normal(size=33333).astype(np.float32),
        "inf": np.where(rng.random(4097) < 0.2, np.inf, rng.random(4097)).astype(np.float32),
        "few_values": rng.integers(0, 4, 100003).astype(np.float32),
        "one": np.array([3.0], dtype=np.float32),
        "large_random": rng.random(1_000_003).astype(np.float32),
        # ties at scale: the tie-break spans hundreds of 4096-element segments
        "zeros_heavy_2m": np.where(rng.random(2_000_017) < 0.7, 0.0,
                                   rng.integers(0, 50, 2_000_017) / 64.0).astype(np.float32),
    }
    for name, s in cases.items():
        for ratio in (0.0, 0.1, 0.5, 0.66, 0.9, 0.9999):
            check_select_exact(torch, ctx, s, ratio)


def test_select_rejects_nan(torch, rb, ctx):
    s = torch.rand(1000, device="cuda")
    s[17] = float("nan")
    with pytest.raises(rb.RefineError) as e:
        ctx.select(s, 0.5)
    assert e.value.status == rb.REFINE_ENONFINITE


def test_nonfinite_and_invalid_inputs(torch, rb, ctx):
    w = synth.random_scene(seed=2, n=500, v=4)
    pos, attr, cams = upload(torch, rb, w.scene, w.cams)
    attr2 = attr.clone()
    attr2[20, 7] = float("inf")
    ctx.score(pos, attr2, cams)
    assert ctx.status() == rb.REFINE_ENONFINITE
    pos2 = pos.clone()
    pos2[1, 3] = float("nan")
    ctx.score(pos2, attr, cams)
    assert ctx.status() == rb.REFINE_ENONFINITE
    bad = w.cams.copy()
    bad[1]["znear"] = -1.0
    ctx.score(pos, attr, rb.cameras_to_device(bad, pos.device))
    assert ctx.status() == rb.REFINE_EINVAL
    attr3 = attr.clone()
    attr3[3:7, 11] = 0.0  # zero quaternion
    ctx.score(pos, attr3, cams)
    assert ctx.status() == rb.REFINE_EINVAL
    assert ctx.status() == rb.REFINE_OK  # reading clears
    # host-side argument checks
    with pytest.raises(rb.RefineError):
        ctx.select(torch.rand(10, device="cuda"), 1.0)
    with pytest.raises(rb.RefineError):
        ctx.score(pos, attr, cams, n_views=0)
    for eta in (0.0, 1e-40):  # zero, and a subnormal float32: the Eq. 17 reciprocal needs eta >= FLT_MIN
        p = rb.default_params(eta=eta)
        with pytest.raises(rb.RefineError):
            ctx.score(pos, attr, cams, params=p)
    # compaction into a too-short output is refused by the device
    s = ctx.score(pos, attr, cams)
    mask, _, nk = ctx.select(s, 0.5)
    ctx.compact(pos, attr, mask, nk, out_row_stride=nk - 1)
    assert ctx.status() == rb.REFINE_EINVAL


def test_deterministic(torch, rb, ctx):
    w = synth.config0(seed=6, n=20000)
    a = gpu_score(torch, rb, ctx, w.scene, w.cams)[0]
    b = gpu_score(torch, rb, ctx, w.scene, w.cams)[0]
    assert np.array_equal(a.view(np.uint32), b.view(np.uint32))


def test_prune_host_matches_device_path(torch, rb, ctx):
    w = synth.config0(seed=7, n=12345)
    s, S, _, (pos, attr) = gpu_score(torch, rb, ctx, w.scene, w.cams)
    mask, thr, nk = ctx.select(torch.from_numpy(s).cuda(), 0.66)
    op, oa, idx = ctx.compact(pos, attr, mask, nk)
    r = ctx.prune_host(torch.from_numpy(w.scene.pos).pin_memory(), torch.from_numpy(w.scene.attr).pin_memory(),
                       w.cams, 0.66, want_scores=True)
    assert r["n_keep"] == nk and r["threshold"] == thr
    assert np.array_equal(r["scores"].numpy().view(np.uint32), s.view(np.uint32))
    assert np.array_equal(r["idx"].numpy(), idx.cpu().numpy())
    assert np.array_equal(r["out_pos"].numpy(), op.cpu().numpy())
    assert np.array_equal(r["out_attr"].numpy(), oa.cpu().numpy())


def test_core_shell_1m_full(torch, rb, ctx):
    """N=1M core-shell scene, 150 hemisphere views at 1297x840: every score
    against the FP64 oracle, masks at the three ratios."""
    w = synth.config1()
    s, S, st, (pos, attr) = gpu_score(torch, rb, ctx, w.scene, w.cams)
    ref = oracle.score(w.scene.params_f64(), w.cams)
    clean = assert_score_parity(s, S, ref)
    assert clean.mean() > 0.97
    np.testing.assert_allclose(st["lambda"], ref["stats"]["lambda"], rtol=1e-6)
    for ratio in w.ratios:
        mask, words, nk = check_select_exact(torch, ctx, s, ratio)
        assert check_mask_vs_oracle_scores(words, ref, ratio, w.scene.n) > 0.999
    check_compact_exact(torch, ctx, w.scene, pos, attr, mask, nk)


@pytest.fixture(scope="module")
def c2_oracle():
    """The FP64 oracle on every primitive of the 3.5M-primitive, 250-view
    benchmark scene (float32 inputs; a few seconds on the host's cores)."""
    w = synth.config2()
    oracle.set_threads(os.cpu_count() or 1)
    return w, oracle.score(w.scene.params_f64(), w.cams)


def test_core_shell_3p5m_full(torch, rb, ctx, c2_oracle):
    """N=3.5M, 250 views at 1600x1063 in the benchmark's launch
    configuration: every score against the FP64 oracle, the keep mask at
    ratio 0.5 against the oracle's own selection outside the threshold band,
    exact selection and compaction of the full scene."""
    w, ref = c2_oracle
    s, S, st, (pos, attr) = gpu_score(torch, rb, ctx, w.scene, w.cams)
    clean = assert_score_parity(s, S, ref)
    assert clean.mean() > 0.97
    np.testing.assert_allclose(st["lambda"], ref["stats"]["lambda"], rtol=1e-6)
    mask, words, nk = check_select_exact(torch, ctx, s, 0.5)
    agree = check_mask_vs_oracle_scores(words, ref, 0.5, w.scene.n)
    print(f"3.5M x 250 FP32: {clean.mean():.4%} of primitives outside the float32 band, "
          f"mask agreement with the oracle {agree:.5%}")
    assert agree > 0.9999
    check_compact_exact(torch, ctx, w.scene, pos, attr, mask, nk)


@pytest.mark.parametrize("dtype,min_agree", [("bf16", 0.999), ("bf16s", 0.9995)])
def test_core_shell_3p5m_bf16_accuracy(torch, rb, ctx, c2_oracle, dtype, min_agree):
    """The precision form on the benchmark scene: rows 3-58 stored as
    bfloat16 (or, for bf16s, rows 6-58 with the log-scales kept float32).
    On its own (rounded) inputs it matches the oracle within the float32
    tolerance (100k-primitive sample); against the oracle on the float32
    scene it was rounded from, the keep mask at ratio 0.5 agrees on at least
    99.9 % of the primitives (99.95 % with float32 log-scales), and the score
    error is reported."""
    w, ref32 = c2_oracle
    sb = w.scene.to_bf16() if dtype == "bf16" else w.scene.to_bf16s()
    s, S, _, _ = gpu_score(torch, rb, ctx, sb, w.cams)
    idx = np.sort(np.random.default_rng(7).choice(w.scene.n, 100_000, replace=False))
    refb = oracle.score_subset(sb.params_f64(), idx, w.cams)
    assert_score_parity(s[idx], S[idx], refb)
    ok = (ref32["nborder"] == 0) & (ref32["scores"] > 0)
    rel = np.abs(s.astype(np.float64)[ok] - ref32["scores"][ok]) / ref32["scores"][ok]
    _, words, _ = check_select_exact(torch, ctx, s, 0.5)
    m_ref, _, _ = oracle.select(ref32["scores"], 0.5)
    agree = float(np.mean(unpack(words, w.scene.n) == unpack(m_ref, w.scene.n)))
    print(f"3.5M x 250 {dtype} vs the FP64 oracle on the float32 scene: rel err mean {rel.mean():.3e} "
          f"p99 {np.quantile(rel, 0.99):.3e} max {rel.max():.3e}; mask agreement {agree:.5%}")
    assert agree >= min_agree


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_padded_row_stride(torch, rb, ctx, dtype):
    """Rows of a scene may be longer than n (row_stride > n): scores,
    selection and compaction equal those of the tightly packed scene."""
    w = synth.random_scene(seed=77, n=12_345, v=20, means="core_shell")
    sc = w.scene.to_bf16() if dtype == "bf16" else w.scene
    dev = torch.device("cuda", 0)
    n, pad = sc.n, 45
    cams = rb.cameras_to_device(w.cams, dev)
    pos = torch.from_numpy(sc.pos).to(dev)
    if dtype == "bf16":
        attr = torch.from_numpy(sc.attr.view(np.int16)).to(dev).view(torch.bfloat16)
    else:
        attr = torch.from_numpy(sc.attr).to(dev)
    pos_p = torch.zeros((3, n + pad), dtype=pos.dtype, device=dev)
    attr_p = torch.zeros((56, n + pad), dtype=attr.dtype, device=dev)
    pos_p[:, :n] = pos
    attr_p[:, :n] = attr
    pos_v, attr_v = pos_p[:, :n], attr_p[:, :n]
    s0 = ctx.score(pos, attr, cams)
    s1 = ctx.score(pos_v, attr_v, cams)
    assert torch.equal(s0, s1)
    m0, thr0, nk = ctx.select(s0, 0.5)
    op0, oa0, i0 = ctx.compact(pos, attr, m0, nk)
    op1, oa1, i1 = ctx.compact(pos_v, attr_v, m0, nk)
    assert torch.equal(i0, i1) and torch.equal(op0, op1) and torch.equal(oa0, oa1)


@pytest.mark.parametrize("dtype,pattern,ratio,pad,opad,with_idx", [
    ("f32", "random", 0.5, 0, 0, True), ("f32", "random", 0.1, 37, 5, True), ("f32", "random", 0.97, 64, 0, True),
    ("f32", "blocks", 0.5, 3, 11, True), ("f32", "random", 0.5, 0, 0, False), ("bf16", "random", 0.66, 9, 2, True),
    ("bf16s", "random", 0.5, 7, 3, True)])
def test_compact_large_ragged(torch, rb, ctx, dtype, pattern, ratio, pad, opad, with_idx):
    """Scenes of about 1.9M primitives or more: FP32 rows are scattered one
    warp per 256-primitive segment, BF16 rows one warp per mask word.  A
    ragged n (not a multiple of 32 or 256), padded input and output rows,
    sparse and dense masks, masks with long all-kept and all-pruned runs, and
    no index output: all bit-exact against the oracle's gather."""
    n = 2_000_003
    rng = np.random.default_rng(4242 + pad)
    pos_h = rng.standard_normal((3, n), dtype=np.float32)
    attr_h = rng.standard_normal((56, n), dtype=np.float32)
    if dtype == "bf16":
        attr_h = synth.f32_to_bf16_bits(attr_h)  # uint16 bit patterns
    elif dtype == "bf16s":
        attr_h[3:] = synth.bf16_bits_to_f32(synth.f32_to_bf16_bits(attr_h[3:]))  # exact in the mixed layout
    scores = rng.random(n, dtype=np.float32)
    if pattern == "blocks":
        scores += ((np.arange(n) // 700) % 3).astype(np.float32)
    dev = torch.device("cuda", 0)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    pos_p = torch.zeros((3, n + pad), dtype=torch.float32, device=dev)
    pos_p[:, :n] = torch.from_numpy(pos_h).to(dev)
    if dtype == "bf16s":
        attr_p = rb.MixedRows.empty(n, stride=n + pad, device=dev)
        attr_p.f32_rows()[:, :n] = torch.from_numpy(attr_h[:3]).to(dev)
        attr_p.bf16_rows()[:, :n] = torch.from_numpy(attr_h[3:]).to(dev).to(torch.bfloat16)
    else:
        attr_p = torch.zeros((56, n + pad), dtype=tdt, device=dev)
    if dtype == "bf16":
        attr_p[:, :n] = torch.from_numpy(attr_h.view(np.int16)).to(dev).view(torch.bfloat16)
    elif dtype == "f32":
        attr_p[:, :n] = torch.from_numpy(attr_h).to(dev)
    m, _, nk = ctx.select(torch.from_numpy(scores).to(dev), ratio)
    op, oa, idx, cnt = ctx.compact(pos_p[:, :n], attr_p[:, :n], m, nk, out_row_stride=nk + opad,
                                   kept_idx=with_idx, return_count=True)
    words = m.cpu().numpy().view(np.uint32)[: (n + 31) // 32]
    kp, ki = oracle.compact(pos_h, words)
    ka, _ = oracle.compact(attr_h, words)
    assert cnt == nk == n - int(np.floor(ratio * n))
    if with_idx:
        assert np.array_equal(idx.cpu().numpy(), ki)
    else:
        assert idx is None
    assert np.array_equal(op[:, :nk].cpu().numpy(), kp[:, :nk])
    got = oa[:, :nk].cpu()
    if dtype == "bf16s":
        got = got.float().numpy()
    else:
        got = got.view(torch.int16).numpy().view(np.uint16) if dtype == "bf16" else got.numpy()
    assert np.array_equal(got, ka[:, :nk])


@pytest.mark.parametrize("v,mv", [(250, 64), (150, 64), (64, 64), (10, 3), (7, 1)])
def test_max_views_subsampling(torch, rb, ctx, v, mv):
    """max_views scores views 0, s, 2s, ... (s = ceil(V / max_views)) with
    |V| their count: the same scores as passing those cameras alone, and
    those agree with the oracle on the subsampled view set."""
    w = synth.random_scene(seed=900 + v, n=20_000, v=v, means="core_shell")
    s = -(-v // mv) if v > mv else 1
    sub = w.cams[::s]
    p = rb.default_params(max_views=mv)
    got, _, _, _ = gpu_score(torch, rb, ctx, w.scene, w.cams, params=p)
    direct, S_direct, _, _ = gpu_score(torch, rb, ctx, w.scene, sub)
    assert np.array_equal(got.view(np.uint32), direct.view(np.uint32))
    ref = oracle.score(w.scene.params_f64(), sub)
    assert_score_parity(direct, S_direct, ref)


def test_max_views_in_batch_and_queue(torch, rb, ctx):
    """The batched form and the request queue apply max_views the same way."""
    w = synth.random_scene(seed=950, n=30_001, v=600, means="core_shell")
    dev = torch.device("cuda", 0)
    p = rb.default_params(max_views=64)
    pos, attr, cd = upload(torch, rb, w.scene, w.cams)
    ref = ctx.score(pos, attr, cd, params=p)
    batch = rb.Batch(ctx, [{"pos": pos, "attr": attr, "cams": cd, "ratio": 0.5}], params=p, compact=False)
    batch.run()
    batch.results()
    assert torch.equal(batch.outputs[0]["scores"], ref)
    batch.close()
    q = rb.Queue(ctx, budget_bytes=2 << 30, max_slots=2, params=p)
    try:
        t = q.submit(w.scene.pos, w.scene.attr, w.cams, 0.5, scores=True)
        res, out = q.poll(t, timeout_ms=60_000)
        assert res["status"] == 0
        assert np.array_equal(np.asarray(out["scores"]).view(np.uint32), ref.cpu().numpy().view(np.uint32))
    finally:
        q.close()


def test_timing_modes(torch, rb, ctx):
    """Kernel timing brackets every launch, or only the score kernel's, and
    reports per-class device times; other modes are refused."""
    w = synth.config0(seed=8)
    dev = torch.device("cuda", 0)
    pos = torch.from_numpy(w.scene.pos).to(dev)
    attr = torch.from_numpy(w.scene.attr).to(dev)
    cams = rb.cameras_to_device(w.cams, dev)
    ctx.kernel_times()
    ctx.set_timing(True, score_only=True)
    s = ctx.score(pos, attr, cams)
    ctx.select(s, 0.5)
    ctx.set_timing(False)
    kt = ctx.kernel_times()
    assert set(kt) == {"score"} and kt["score"]["launches"] == 1 and kt["score"]["ms"] > 0
    ctx.set_timing(True)
    s = ctx.score(pos, attr, cams)
    ctx.select(s, 0.5)
    ctx.set_timing(False)
    kt = ctx.kernel_times()
    assert {"features", "score", "select_mask"} <= set(kt) and all(v["ms"] > 0 for v in kt.values())
    assert rb.refine_ctx_set_timing(ctx.handle, 3) == rb.REFINE_EINVAL


@pytest.mark.parametrize("n,v,flags", [(63, 65, 0), (64, 96, 0), (65, 129, 0), (3000, 64, 0), (3000, 65, 0), (40_001, 577, 0),
                                       (40_001, 130, 1 << 4), (320_000, 66, 0)])
def test_split_tiles_same_bits(torch, rb, ctx, n, v, flags):
    """Tiles whose views are split into items (the plain call) against whole
    tiles (the counting call, which splits none): the same bits, for view
    counts about the item and block sizes, one and two passes, more tiles
    than one wave, a tile holding an underflowed scale, and repeated calls."""
    w = synth.random_scene(seed=n + v, n=n, v=v, means="core_shell")
    w.scene.attr[0, n // 2] = -200.0
    if flags:
        w.cams["znear"] = 1.0
    pos, attr, cams = upload(torch, rb, w.scene, w.cams)
    p = rb.default_params(flags=rb.FLAG_NORM_ATTR | flags)
    whole, _ = ctx.score(pos, attr, cams, params=p, stats=True)
    for _ in range(2):
        vs = torch.empty(n, dtype=torch.float32, device=pos.device)
        split = ctx.score(pos, attr, cams, params=p, view_sum=vs)
        assert torch.equal(split.view(torch.int32), whole.view(torch.int32))
    if n <= 3000:
        ref = oracle.score(w.scene.params_f64(), w.cams, oracle_params_from(p, rb))
        assert_score_parity(split.cpu().numpy(), vs.cpu().numpy(), ref)


@pytest.mark.parametrize("n", [1, 31, 33, 6_144, 6_145, 12_289, 24_577, 49_152, 49_153, 131_072, 131_073, 262_144, 262_145])
def test_select_cluster_edges(torch, rb, ctx, n):
    """Sizes about the cluster selection's CTA counts, range ends and limit,
    with ties that span CTAs, all scores equal, and an unaligned score
    pointer: bit-exact against the oracle."""
    rng = np.random.default_rng(n)
    for s in (rng.random(n), rng.integers(0, 3, n) / 4.0, np.full(n, -2.5), np.sort(rng.random(n))[::-1]):
        s = np.ascontiguousarray(s, dtype=np.float32)
        for ratio in (0.1, 0.5, 0.9999):
            check_select_exact(torch, ctx, s, ratio)
    t = torch.from_numpy(np.concatenate([[9.0], s]).astype(np.float32)).cuda()[1:]
    mask, thr, nk = ctx.select(t, 0.66)
    m_ref, thr_ref, nk_ref = oracle.select(s.astype(np.float64), 0.66)
    assert nk == nk_ref and thr == np.float32(thr_ref)
    assert np.array_equal(mask.cpu().numpy().view(np.uint32)[: (n + 31) // 32], m_ref)
    # the entry point whose kernels are not chained takes the cluster form up to its own limit
    s = (rng.integers(0, 3, n) / 4.0).astype(np.float32)
    t = torch.from_numpy(s).cuda()
    m2 = torch.empty((n + 31) // 32, dtype=torch.int32, device="cuda")
    c_thr, err = ctypes.c_float(), ctypes.create_string_buffer(64)
    st = rb.refine_select_noalloc(t.data_ptr(), n, 0.66, m2.data_ptr(), ctypes.byref(c_thr), None, err, 64,
                                  torch.cuda.current_stream().cuda_stream)
    m_ref, thr_ref, _ = oracle.select(s.astype(np.float64), 0.66)
    assert st == rb.REFINE_OK and c_thr.value == (np.float32(thr_ref) if n > 1 else -math.inf)
    assert np.array_equal(m2.cpu().numpy().view(np.uint32), m_ref)


@pytest.mark.parametrize("n", [255, 256, 257, 65_536, 65_537, 1_048_577, 16_777_216, 16_777_217])
def test_compact_count_sizes(torch, rb, ctx, n):
    """Kept counts and offsets about the segment, block and size limits of the
    counting kernels, checked through the indices (the attribute rows are zeros)."""
    g = torch.Generator(device="cuda").manual_seed(n)
    keep = torch.rand(n, generator=g, device="cuda") < 0.03
    words = (n + 31) // 32
    bits = torch.zeros(words * 32, dtype=torch.int64, device="cuda")
    bits[:n] = keep
    w = (bits.view(words, 32) << torch.arange(32, device="cuda")).sum(1)
    mask = w.to(torch.int32) if n % 2 else torch.cat([w[:1], w]).to(torch.int32)[1:]  # both alignments
    pos = torch.arange(n, device="cuda", dtype=torch.float32).repeat(3, 1)
    attr = torch.zeros((56, n), device="cuda", dtype=torch.bfloat16)
    want = torch.nonzero(keep).flatten().to(torch.int32)
    op, oa, idx, cnt = ctx.compact(pos, attr, mask, want.numel(), return_count=True)
    assert cnt == want.numel() and torch.equal(idx, want) and torch.equal(op[2], pos[2][want.long()])
    ctx.check()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "bf16s"])
@pytest.mark.parametrize("pad", [0, 1, 3, 6])
def test_compact_units(torch, rb, ctx, dtype, pad):
    """The scatter about its units (128 or 256 primitives) and the end of a
    scene, with row strides of every 16-byte misalignment: equal to indexing
    the rows."""
    for n in (1, 7, 8, 127, 128, 129, 136, 137, 255, 256, 257, 263, 264, 265, 385, 1_031, 70_003):
        g = torch.Generator(device="cuda").manual_seed(n * 10 + pad)
        S = n + pad
        pos = torch.randn((3, S), generator=g, device="cuda")
        full = torch.randn((56, S), generator=g, device="cuda")
        for p in (0.02, 0.5, 1.0):
            keep = torch.rand(n, generator=g, device="cuda") < p
            words = (n + 31) // 32
            bits = torch.zeros(words * 32, dtype=torch.int64, device="cuda")
            bits[:n] = keep
            mask = (bits.view(words, 32) << torch.arange(32, device="cuda")).sum(1).to(torch.int32)
            want = torch.nonzero(keep).flatten()
            if dtype == "bf16s":
                attr = rb.MixedRows.from_float(full)  # stride S
                attr = attr.to("cuda")[:, :n]
                rows = attr.float()
            else:
                attr = full.to(torch.bfloat16 if dtype == "bf16" else torch.float32)[:, :n]
                rows = attr.float()
            op, oa, idx = ctx.compact(pos[:, :n], attr, mask, want.numel(), out_row_stride=want.numel() + 1 + pad)
            assert torch.equal(idx, want.to(torch.int32))
            assert torch.equal(op, pos[:, want]), (n, p)
            assert torch.equal(oa.float().to("cuda"), rows[:, want].to("cuda")), (n, p)
    ctx.check()


@pytest.mark.parametrize("n,v,dtype", [(900, 5, "f32"), (20_001, 33, "bf16"), (300_007, 70, "bf16s"), (270_000, 20, "f32")])
def test_chained_calls_same_bits(torch, rb, ctx, n, v, dtype):
    """The plain calls, whose kernels overlap their launches, one after another
    on two scenes in turn without a wait in between, and captured in a graph:
    the same bits as the batched form, whose kernels do not."""
    scenes, want = [], []
    for k in range(2):
        w = synth.random_scene(seed=n + k, n=n - 7 * k, v=v, means="core_shell")
        sc = w.scene if dtype == "f32" else (w.scene.to_bf16() if dtype == "bf16" else w.scene.to_bf16s())
        pos, attr, cams = upload(torch, rb, sc, w.cams)
        scenes.append((pos, attr, cams))
        b = rb.Batch(ctx, [{"pos": pos, "attr": attr, "cams": cams, "ratio": 0.6}])
        b.run()
        b.results()
        want.append({x: (y if isinstance(y, int) else y.float().cpu() if x == "out_attr" else y.clone())
                     for x, y in b.outputs[0].items()})
        b.close()

    def one(k):
        pos, attr, cams = scenes[k]
        s = ctx.score(pos, attr, cams)
        mask, _, nk = ctx.select(s, 0.6, threshold=False)
        return (s, mask) + ctx.compact(pos, attr, mask, nk)

    def same(k, got):
        s, mask, op, oa, idx = got
        return (torch.equal(s, want[k]["scores"]) and torch.equal(mask, want[k]["mask"]) and torch.equal(op, want[k]["out_pos"])
                and torch.equal(oa.float().cpu(), want[k]["out_attr"]) and torch.equal(idx, want[k]["idx"]))
    got = [(i % 2, one(i % 2)) for i in range(24)]
    torch.cuda.synchronize()
    assert all(same(k, g) for k, g in got)
    ctx.check()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        one(0), one(1)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            held = [one(0), one(1)]
        for _ in range(3):
            graph.replay()
        stream.synchronize()
        assert all(same(k, held[k]) for k in range(2))
        ctx.check()


@pytest.mark.parametrize("scale", [0.5, 1.0, 1.5])
def test_scaled_world_to_camera(torch, rb, ctx, scale):
    """World-to-camera rows that are not orthonormal (a scale in the extrinsics)
    get no footprint bound: scores against the oracle, which forms J W Sigma
    W^T J^T as it stands."""
    w = synth.random_scene(seed=31, n=5000, v=20, means="core_shell")
    w.cams["R"] *= np.float32(scale)
    w.cams["t"] *= np.float32(scale)
    s, S, _, _ = gpu_score(torch, rb, ctx, w.scene, w.cams)
    assert_score_parity(s, S, oracle.score(w.scene.params_f64(), w.cams))


@pytest.mark.parametrize("v", [306, 333, 335, 384, 385, 512])
def test_camera_block_shared_memory(torch, rb, ctx, v):
    """Camera blocks about the 48 KB of shared memory that a launch gets
    without opting in (static part included), for Eq. 17 and for the longer
    records of FULL_JACOBIAN: plain, counting and batched launches."""
    w = synth.config0(seed=6, n=700)
    cams = np.resize(w.cams, v)
    cams["znear"] = 1.0  # (as in test_ablation_flags)
    for flags in (rb.FLAG_NORM_ATTR, rb.FLAG_NORM_ATTR | rb.FLAG_FULL_JACOBIAN):
        p = rb.default_params(flags=flags)
        s, S, _, (pos, attr) = gpu_score(torch, rb, ctx, w.scene, cams, params=p)
        assert_score_parity(s, S, oracle.score(w.scene.params_f64(), cams, oracle_params_from(p, rb)))
        cd = rb.cameras_to_device(cams, pos.device)
        plain = ctx.score(pos, attr, cd, params=p)
        assert np.array_equal(plain.cpu().numpy(), s)
        batch = rb.Batch(ctx, [{"pos": pos, "attr": attr, "cams": cd, "ratio": 0.5}], params=p)
        batch.run()
        batch.results()
        assert torch.equal(batch.outputs[0]["scores"], plain)
        batch.close()


def test_select_threads_of_two_sizes(torch, rb):
    """Two threads, each with a context and a stream, select from different
    sizes at once: one's launch settings do not disturb the other's."""
    import threading
    failed = []
    scores = {n: np.random.default_rng(n).random(n).astype(np.float32) for n in (50_000, 120_000)}
    refs = {n: oracle.select(s.astype(np.float64), 0.5) for n, s in scores.items()}  # (one at a time)

    def work(n):
        try:
            c, s = rb.Context(0), torch.cuda.Stream()
            t = torch.from_numpy(scores[n]).cuda()
            mask = torch.empty((n + 31) // 32, dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            for _ in range(400):
                _, _, nk = c.select(t, 0.5, mask=mask, threshold=False, stream=s)
            s.synchronize()
            m_ref, _, nk_ref = refs[n]
            assert nk == nk_ref and np.array_equal(mask.cpu().numpy().view(np.uint32), m_ref)
            c.close()
        except Exception as e:  # noqa: BLE001 -- reported below
            failed.append((n, repr(e)))

    threads = [threading.Thread(target=work, args=(n,)) for n in scores]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
