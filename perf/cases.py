"""Performance cases: the work that a user of this package has it do, through
its public entry points (``binding.Context``, ``Batch`` and ``Queue``).

Every case is a dict of plain values; its ``kind`` says which calls it makes:

  prune    score + select + compact of one device-resident scene, the three
           plain calls that a training loop makes to prune its scene
  reprune  select + compact at three ratios of scores that are already there
           (looking for the ratio to use)
  batch    many scenes of uneven size in one ``Batch`` run
  serve    pruning requests for host-resident scenes through a ``Queue``
  host     ``Context.prune_host``: one scene from page-locked host memory

Scenes follow the recipes of ``synth.py`` (the same distributions, drawn on
the GPU from the seed) and the cameras come from that module.
"""
import math

import numpy as np
import torch

from paper_2606_09074_gb300 import binding as rb
from paper_2606_09074_gb300 import synth

RES = synth.RESOLUTIONS  # 960x540, 1297x840, 1600x1063


def listed():
    return [
        # The small scene of the tests: where launches and latency count.
        dict(name="small_f32", kind="prune", n=10_000, v=16, w=640, h=480, focal=512.0, means="normal2", rig="ring",
             dtype="f32", ratio=0.5, max_views=0, flags="default"),
        # An object-sized scene of odd size (rows not 16-byte aligned to one another) in the mixed storage.
        dict(name="ragged_bf16s", kind="prune", n=77_773, v=61, w=960, h=540, focal=1100.0, means="core_shell",
             rig="hemisphere", dtype="bf16s", ratio=0.66, max_views=0, flags="default"),
        # An ordinary scene: 1M primitives, 150 training views.
        dict(name="medium_f32", kind="prune", n=1_000_000, v=150, w=1297, h=840, focal=1100.0, means="core_shell",
             rig="hemisphere", dtype="f32", ratio=0.66, max_views=0, flags="default"),
        # The benchmark's scene, in float32 and in bfloat16 storage.
        dict(name="large_f32", kind="prune", n=3_500_000, v=250, w=1600, h=1063, focal=1100.0, means="core_shell",
             rig="hemisphere", dtype="f32", ratio=0.5, max_views=0, flags="default"),
        dict(name="large_bf16", kind="prune", n=3_500_000, v=250, w=1600, h=1063, focal=1100.0, means="core_shell",
             rig="hemisphere", dtype="bf16", ratio=0.5, max_views=0, flags="default"),
        # The paper's own setting: 64 of the views scored, an odd number of primitives.
        dict(name="views64_f32", kind="prune", n=1_750_001, v=300, w=1600, h=1063, focal=1100.0, means="core_shell",
             rig="hemisphere", dtype="f32", ratio=0.5, max_views=64, flags="default"),
        # A long capture: more views than one camera block holds.
        dict(name="many_views_f32", kind="prune", n=150_000, v=1100, w=1297, h=840, focal=1100.0, means="core_shell",
             rig="hemisphere", dtype="f32", ratio=0.9, max_views=0, flags="default"),
        # Choosing a ratio: the three ratios of the tests on scores that are there.
        dict(name="reprune_f32", kind="reprune", n=1_000_000, dtype="f32", zeros=0.05),
        # Twelve scenes of the batching workload (its first seeds' sizes), bfloat16.
        dict(name="batch12_bf16", kind="batch", scenes=12, spec=100, nmin=50_000, nmax=2_000_000, dtype="bf16", ratio=0.66),
        # Eight jobs of the serving workload (its first seeds' sizes and ratios), bfloat16, from host memory.
        dict(name="serve8_bf16", kind="serve", jobs=8, spec=1000, nmin=50_000, nmax=3_500_000, dtype="bf16"),
        # One ordinary scene pruned from host memory to host memory.
        dict(name="host_f32", kind="host", n=1_000_000, v=150, w=1297, h=840, focal=1100.0, means="core_shell",
             rig="hemisphere", dtype="f32", ratio=0.5, max_views=0, flags="default"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("prune", "reprune", "batch", "serve", "host"), weights=(8, 2, 2, 1, 1))[0]
    dtype = rng.choice(("f32", "f32", "bf16", "bf16s"))
    if kind == "reprune":
        return dict(kind=kind, n=_log_uniform(rng, 2_000, 3_500_000), dtype=dtype, zeros=rng.choice((0.0, 0.05, 0.3, 0.7)))
    if kind == "batch":
        # a scene count and a largest size that stay below the listed batch's work
        scenes = rng.randint(2, 12)
        return dict(kind=kind, scenes=scenes, spec=rng.randint(164, 9_999), nmin=10_000, nmax=_log_uniform(rng, 60_000, 800_000),
                    dtype=dtype, ratio=rng.choice((0.5, 0.66, 0.9)))
    if kind == "serve":
        return dict(kind=kind, jobs=rng.randint(2, 8), spec=rng.randint(1_010, 2_990), nmin=50_000, nmax=250_000,
                    dtype=rng.choice(("bf16", "bf16s")))
    n = _log_uniform(rng, 1_000, 3_500_000 if kind == "prune" else 1_000_000)
    most = min(1_500 if kind == "prune" else 300, 875_000_000 // n)
    v = min(_log_uniform(rng, 8, most), most)
    w, h = rng.choice(RES)
    return dict(kind=kind, n=n, v=v, w=w, h=h, focal=1100.0, means=rng.choice(("core_shell", "core_shell", "normal2")),
                rig=rng.choice(("hemisphere", "hemisphere", "ring")), dtype=dtype, ratio=rng.choice((0.3, 0.5, 0.66, 0.9)),
                max_views=rng.choice((0, 0, 0, 64)),
                flags=rng.choice(("default", "default", "default", "default", "no_vis", "no_proj", "equal_lambda")))


# ------------------------------------------------------------------ inputs

def _sizes(case, k):
    """(n, views, (width, height), ratio) of scene k of a batch or serving case, as synth's recipes draw them."""
    rng = np.random.default_rng(case["spec"] + k)
    n = int(round(math.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"])))))
    v = int(rng.integers(50, 301))
    wh = RES[int(rng.integers(0, len(RES)))]
    ratio = (0.5, 0.66, 0.9)[int(rng.integers(0, 3))] if case["kind"] == "serve" else case["ratio"]
    return n, v, wh, ratio


def _rows(n, means, seed):
    """pos [3, n] and attr [56, n] float32 on the GPU, by the distributions of synth.py."""
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev)
    g.manual_seed(seed)

    def normal(rows):
        return torch.randn((rows, n), generator=g, device=dev)

    def uniform(lo, hi):
        return lo + (hi - lo) * torch.rand(n, generator=g, device=dev)

    if means == "normal2":
        pos = (2.0 * normal(3)).clamp_(-6.0, 6.0)
    else:
        core = uniform(0.0, 1.0) < 0.7
        mid, d = 1.5 * normal(3), normal(3)
        d /= d.norm(dim=0, keepdim=True).clamp_min(1e-12)
        pos = torch.where(core, mid, d * uniform(6.0, 10.0)).contiguous()
    attr = torch.empty((56, n), device=dev)
    attr[0:3] = normal(3) - 4.5
    q = normal(4)
    attr[3:7] = q / q.norm(dim=0, keepdim=True).clamp_min(1e-12)
    attr[7] = 2.0 * normal(1)[0]
    attr[8:11] = 0.5 * normal(3)
    attr[11:56] = 0.1 * normal(45)
    return pos, attr


def _stored(attr, dtype):
    if dtype == "bf16":
        return attr.to(torch.bfloat16)
    if dtype == "bf16s":
        return rb.MixedRows.from_float(attr, device=attr.device)
    return attr


def _cams(v, w, h, focal, rig, seed):
    centers = (synth.ring_centers(v) if rig == "ring"
               else synth.hemisphere_centers(np.random.default_rng(seed), v))
    return synth.make_cameras(centers, w, h, focal)


def _one(case, seed):
    pos, attr = _rows(case["n"], case["means"], seed)
    return pos, attr, _cams(case["v"], case["w"], case["h"], case["focal"], case["rig"], seed)


def _of_many(case, k, seed):
    """Scene k of a batch or serving case."""
    n, v, wh, ratio = _sizes(case, k)
    s = seed * 1009 + k
    pos, attr = _rows(n, "core_shell", s)
    return pos, attr, _cams(v, wh[0], wh[1], 1100.0, "hemisphere", s), ratio


def _params(case):
    flags = rb.FLAG_NORM_ATTR | {"default": 0, "no_vis": rb.FLAG_NO_VIS, "no_proj": rb.FLAG_NO_PROJ,
                                 "equal_lambda": rb.FLAG_EQUAL_LAMBDA}[case["flags"]]
    return rb.default_params(flags=flags, max_views=case["max_views"])


_kept = {}


def _context():
    # one context for the life of the program, as a user's program keeps
    if "ctx" not in _kept:
        _kept["ctx"] = rb.Context(0)
    return _kept["ctx"]


def _queue():
    # one queue for the life of the program, as a server keeps
    if "queue" not in _kept:
        _kept["queue"] = rb.Queue(_context(), budget_bytes=16 << 30, max_slots=8)
    return _kept["queue"]


def _pinned(attr, dtype):
    a = _stored(attr, dtype)
    if dtype == "bf16s":
        out = rb.MixedRows.empty(a.n, pin_memory=True)
        out.buf.copy_(a.buf)
        return out
    return torch.empty(a.shape, dtype=a.dtype, pin_memory=True).copy_(a)


def _host_outputs(attr, n_keep):
    return {"out_pos": torch.empty((3, n_keep), dtype=torch.float32, pin_memory=True),
            "out_attr": rb.empty_attr_like(attr, n_keep, pin_memory=True),
            "idx": torch.empty(n_keep, dtype=torch.int32, pin_memory=True)}


def _scores(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 77)
    s = torch.exp(2.0 * torch.randn(case["n"], generator=g, device="cuda") - 3.0)
    s[torch.rand(case["n"], generator=g, device="cuda") < case["zeros"]] = 0.0
    return s


def prepare(case, seed):
    kind = case["kind"]
    ctx = _context()
    if kind == "prune":
        pos, attr, cams = _one(case, seed)
        return {"kind": kind, "ctx": ctx, "pos": pos, "attr": _stored(attr, case["dtype"]),
                "cams": rb.cameras_to_device(cams, pos.device), "ratio": case["ratio"], "params": _params(case)}
    if kind == "reprune":
        pos, attr = _rows(case["n"], "core_shell", seed)
        return {"kind": kind, "ctx": ctx, "pos": pos, "attr": _stored(attr, case["dtype"]), "scores": _scores(case, seed)}
    if kind == "batch":
        jobs = []
        for k in range(case["scenes"]):
            pos, attr, cams, ratio = _of_many(case, k, seed)
            jobs.append({"pos": pos, "attr": _stored(attr, case["dtype"]), "cams": rb.cameras_to_device(cams, pos.device),
                         "ratio": ratio})
        return {"kind": kind, "batch": rb.Batch(ctx, jobs)}
    if kind == "serve":
        jobs = []
        for k in range(case["jobs"]):
            pos, attr, cams, ratio = _of_many(case, k, seed)
            attr_h = _pinned(attr, case["dtype"])
            n = pos.shape[1]
            out = _host_outputs(attr_h, n - int(math.floor(ratio * n)))
            out["mask"] = torch.empty((n + 31) // 32, dtype=torch.int32, pin_memory=True)
            jobs.append((torch.empty(pos.shape, pin_memory=True).copy_(pos), attr_h, cams, ratio, out))
        return {"kind": kind, "queue": _queue(), "jobs": jobs}
    pos, attr, cams = _one(case, seed)
    attr_h = _pinned(attr, case["dtype"])
    out = _host_outputs(attr_h, case["n"] - int(math.floor(case["ratio"] * case["n"])))
    return {"kind": kind, "ctx": ctx, "pos": torch.empty(pos.shape, pin_memory=True).copy_(pos), "attr": attr_h, "cams": cams,
            "ratio": case["ratio"], "params": _params(case), "out": out}


def _tensors(attr):
    """The rows of an attribute block as tensors."""
    if isinstance(attr, rb.MixedRows):
        return [attr.f32_rows()[:, : attr.n], attr.bf16_rows()[:, : attr.n]]
    return attr


def run(state):
    kind = state["kind"]
    if kind == "prune":
        ctx = state["ctx"]
        scores = ctx.score(state["pos"], state["attr"], state["cams"], params=state["params"])
        mask, _, n_keep = ctx.select(scores, state["ratio"], threshold=False)
        pos, attr, idx = ctx.compact(state["pos"], state["attr"], mask, n_keep)
        return {"scores": scores, "mask": mask, "pos": pos, "attr": _tensors(attr), "idx": idx}
    if kind == "reprune":
        ctx, got = state["ctx"], []
        for ratio in (0.5, 0.66, 0.9):
            mask, _, n_keep = ctx.select(state["scores"], ratio, threshold=False)
            pos, attr, idx = ctx.compact(state["pos"], state["attr"], mask, n_keep)
            got.append({"mask": mask, "pos": pos, "attr": _tensors(attr), "idx": idx})
        return got
    if kind == "batch":
        state["batch"].run()
        return [{"scores": o["scores"], "mask": o["mask"], "pos": o["out_pos"], "attr": _whole(o["out_attr"]), "idx": o["idx"]}
                for o in state["batch"].outputs]
    if kind == "serve":
        q = state["queue"]
        tickets = [q.submit(pos, attr, cams, ratio, outputs=out) for pos, attr, cams, ratio, out in state["jobs"]]
        got = []
        for t in tickets:
            res, out = q.poll(t)
            if res["status"] != rb.REFINE_OK:
                raise RuntimeError(f"request failed with status {res['status']}")
            got.append({"threshold": res["threshold"], "mask": out["mask"], "pos": out["out_pos"],
                        "attr": _whole(out["out_attr"]), "idx": out["idx"]})
        return got
    r = state["ctx"].prune_host(state["pos"], state["attr"], state["cams"], state["ratio"], params=state["params"],
                                out=state["out"])
    return {"threshold": r["threshold"], "n_keep": r["n_keep"], "pos": r["out_pos"], "attr": _tensors(r["out_attr"]),
            "idx": r["idx"]}


def _whole(attr):
    return attr.buf if isinstance(attr, rb.MixedRows) else attr


# -------------------------------------------------------------------- work

_COL = {"f32": 224, "bf16": 112, "bf16s": 118}  # bytes of the 56 attribute rows per primitive


def _scored_views(v, max_views):
    step = -(-v // max_views) if 0 < max_views < v else 1
    return -(-v // step)


def _prune_work(n, v, dtype, ratio, scored):
    n_keep = n - int(math.floor(ratio * n))
    col = 12 + _COL[dtype]
    # the scene and the cameras in; scores, mask, kept rows and indices out.  A visible pair needs its
    # depth (6), z^2 + eta (2), the reciprocal and the add.
    return {"bytes": n * col + 80 * v + 4 * n + n // 8 + n_keep * (col + 4), "flops": 10 * n * scored}


def work(case):
    kind = case["kind"]
    if kind in ("prune", "host"):
        return _prune_work(case["n"], case["v"], case["dtype"], case["ratio"], _scored_views(case["v"], case["max_views"]))
    if kind == "reprune":
        n, col = case["n"], 12 + _COL[case["dtype"]]
        keep = [n - int(math.floor(r * n)) for r in (0.5, 0.66, 0.9)]
        # the scores and the scene read once, a mask and the kept rows and indices of each ratio written
        return {"bytes": n * (col + 4) + 3 * (n // 8) + sum(keep) * (col + 4), "flops": 3 * n}
    total = {"bytes": 0, "flops": 0}
    for k in range(case["scenes"] if kind == "batch" else case["jobs"]):
        n, v, _, ratio = _sizes(case, k)
        one = _prune_work(n, v, case["dtype"], ratio, v)
        total = {key: total[key] + one[key] for key in total}
    return total


# ------------------------------------------------------------------- exact

def _exact_scores(pos, attr, cams, max_views, flags, dtype):
    """Scores in 64 bits from the paper's formulas (Eq. 1, 7, 13-14, 17-20), plain torch."""
    if dtype == "bf16":
        attr = attr.to(torch.bfloat16).float()
    elif dtype == "bf16s":
        attr = torch.cat([attr[:3], attr[3:].to(torch.bfloat16).float()])
    mu, a = pos.double(), attr.double()
    n = mu.shape[1]
    eta = float(np.float32(0.05))
    p = rb.default_params()
    luma = [float(x) for x in p.luma]
    s = torch.exp(a[0:3])
    w, x, y, z = a[3:7] / a[3:7].norm(dim=0, keepdim=True)
    alpha = torch.sigmoid(a[7])
    rot = [[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
           [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
           [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]]
    cov = {}
    for i in range(3):
        for j in range(i, 3):
            cov[i, j] = sum(rot[i][k] * rot[j][k] * s[k] * s[k] for k in range(3))
            cov[j, i] = cov[i, j]
    del rot
    # content features (variance of the luma of the DC colour, mean of alpha (1 - alpha), mean scale ratio)
    lum = sum(luma[k] * a[8 + k] for k in range(3)) * (0.5 / math.sqrt(math.pi))
    f_col = float((lum - lum.mean()).square().mean())
    f_opa = float((alpha * (1 - alpha)).mean())
    order = torch.sort(s, dim=0).values
    f_gem = float((order[2] / (order[0] + eta)).mean())
    lam = [max(v, 0.0) for v in (math.log(f_gem + eta) / p.e_ln_gem, f_col / p.e_col, f_opa / p.e_opa)]
    lam = [v / sum(lam) for v in lam] if sum(lam) > 0 and flags != "equal_lambda" else [1 / 3] * 3
    mags = [order[2] * order[1], a[8:56].norm(dim=0), alpha]
    coupled = sum(l / float(m.mean()) * m for l, m in zip(lam, mags) if float(m.mean()) > 0)
    del a, order, lum
    step = -(-len(cams) // max_views) if 0 < max_views < len(cams) else 1
    cams = cams[::step]
    total = torch.zeros(n, dtype=torch.float64, device=mu.device)
    for c in cams:
        R, t = c["R"].astype(np.float64).reshape(3, 3), c["t"].astype(np.float64)
        fx, fy, cx, cy = (float(c[k]) for k in ("fx", "fy", "cx", "cy"))
        px, py, pz = (R[i, 0] * mu[0] + R[i, 1] * mu[1] + R[i, 2] * mu[2] + t[i] for i in range(3))
        vis = (pz > float(c["znear"])) & (pz < float(c["zfar"]))
        for f, off, row, q, size in ((fx, cx, R[0], px, float(c["width"])), (fy, cy, R[1], py, float(c["height"]))):
            centre = f * q / pz + off
            # the row of J W: f (row / z - q R2 / z^2)
            j = [f / pz * (row[k] - q / pz * R[2, k]) for k in range(3)]
            var = sum(j[i] * j[k] * cov[i, k] * (1 if i == k else 2) for i in range(3) for k in range(i, 3))
            r = 3 * torch.sqrt(var.clamp_min_(0.0))
            vis &= (centre + r >= 0) & (centre - r <= size)
        total += torch.where(vis, torch.ones_like(pz) if flags == "no_proj" else 1 / (pz * pz + eta), torch.zeros_like(pz))
    return (torch.ones_like(alpha) if flags == "no_vis" else alpha) * total / len(cams) * coupled


def _exact_threshold(scores, ratio):
    n = scores.numel()
    cut = int(math.floor(ratio * n))
    return float(torch.sort(scores).values[cut]) if cut else -math.inf


def exact(case, seed):
    kind = case["kind"]
    if kind == "prune":
        pos, attr, cams = _one(case, seed)
        s = _exact_scores(pos, attr, cams, case["max_views"], case["flags"], case["dtype"])
        return {"scores": s, "mask": None, "pos": None, "attr": None, "idx": None}
    if kind == "host":
        pos, attr, cams = _one(case, seed)
        s = _exact_scores(pos, attr, cams, case["max_views"], case["flags"], case["dtype"])
        return {"threshold": _exact_threshold(s, case["ratio"]), "n_keep": None, "pos": None, "attr": None, "idx": None}
    if kind == "reprune":
        return None  # masks and moved rows: compared value for value
    got = []
    for k in range(case["scenes"] if kind == "batch" else case["jobs"]):
        pos, attr, cams, ratio = _of_many(case, k, seed)
        s = _exact_scores(pos, attr, cams, 0, "default", case["dtype"])
        key, value = ("scores", s) if kind == "batch" else ("threshold", _exact_threshold(s, ratio))
        got.append({key: value, "mask": None, "pos": None, "attr": None, "idx": None})
    return got
