"""Performance cases: the renders a user of this library has it do, through the
public entry points of the binding, from an interactive preview to a batch of
full-HD frames.

A case is a dict of plain values; ``prepare(case, seed)`` makes its scenes (the
Julia constants and slice frames come from the seed) and output planes,
``run(state)`` is one pass, ``work(case)`` its unavoidable bytes and flops, and
``exact(case, seed)`` what the pass returns for its real-valued planes, in plain
FP64 torch.
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2303_14827_gb300 import binding, scenes

PRECISION = {"fp32": scenes.PRECISION_FP32, "recheck": scenes.PRECISION_FP32_RECHECK, "fp64": scenes.PRECISION_FP64}
TRAVERSAL = {"march": scenes.TRAVERSAL_MARCH, "de": scenes.TRAVERSAL_DE}
PLANES = ("iter", "depth", "normal", "rgba")


def _case(name, kind, width, height, **kw):
    c = {"name": name, "kind": kind, "width": width, "height": height, "frames": 1, "precision": "recheck",
         "traversal": "march", "c": "uniform", "slice": "axis", "modulus": 0, "square": 0, "max_iter": 16,
         "march_steps": 512, "bisect_steps": 10, "grid": 0}
    c.update(kw)
    return c


def listed() -> list:
    return [
        # the single small frame of the paper's standard view: an interactive
        # preview, where launches and latency count
        _case("preview_256", "render", 256, 256, precision="fp32", c="walk", max_iter=12, march_steps=256,
              bisect_steps=8),
        # one frame of an exploration session at contract accuracy, ragged size,
        # with many hit pixels and long orbits
        _case("explore_701x509", "render", 701, 509, c="walk", max_iter=24),
        # full HD without the FP64 recheck: the fast preview of a still
        _case("full_hd_fp32", "render", 1920, 1080, precision="fp32"),
        # full HD still of the paper's caption constants at contract accuracy:
        # hundreds of thousands of hit pixels
        _case("full_hd_paper", "render", 1920, 1080, c="paper", max_iter=15),
        # five full-HD frames in one call: offline rendering of a sequence, the
        # benchmark's headline workload
        _case("full_hd_batch5", "batch", 1920, 1080, frames=5),
        # a random 3-D slice of the 8-D set, all eight components in play
        _case("slice_1024", "render", 1024, 1024, slice="random", max_iter=20),
        # the all-FP64 mode: ground truth for a still, odd size
        _case("fp64_481x271", "render", 481, 271, precision="fp64", c="walk"),
        # sphere tracing (the paper's own traversal), fast and contract-accurate
        _case("de_full_hd_fp32", "render", 1920, 1080, precision="fp32", traversal="de"),
        _case("de_full_hd", "render", 1920, 1080, traversal="de", c="walk"),
        # a dense occupancy grid (the paper's voxel figure, at its finest here)
        _case("voxels_1024", "voxelize", 16, 16, precision="fp32", c="walk", grid=1024),
        # the image of a grid, beside the ray-traced one in the paper's figure
        _case("voxel_image_200", "voxel_image", 1920, 1080, c="walk", grid=200),
        # a burst of served requests of mixed sizes, submitted and polled
        _case("served_16", "served", 1024, 1024, frames=16, c="walk"),
    ]


def _log_int(rng, lo, hi):
    return int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))


def draw(rng) -> dict:
    """One more case of the same ranges; no more pixels, samples or cells than
    the largest listed case of its kind."""
    kind = rng.choice(["render"] * 6 + ["batch", "host", "voxelize", "voxel_image", "served"])
    width, height = _log_int(rng, 64, 1920), _log_int(rng, 64, 1080)
    kw = {"precision": rng.choice(["fp32", "recheck", "recheck"]), "c": rng.choice(["uniform", "walk", "paper"]),
          "slice": rng.choice(["axis", "axis", "random"]), "max_iter": rng.randint(6, 32),
          "march_steps": _log_int(rng, 96, 512), "bisect_steps": rng.randint(4, 10)}
    if kind == "render":
        kw["traversal"] = rng.choice(["march", "march", "march", "de"])
        kw["modulus"] = rng.choice([0, 0, 0, 1])
        kw["square"] = rng.choice([0, 0, 0, 1])
        if kw["traversal"] == "march" and rng.random() < 0.2:
            kw["precision"] = "fp64"
            width, height = _log_int(rng, 64, 481), _log_int(rng, 64, 271)
    elif kind in ("batch", "host"):
        kw["frames"] = rng.randint(2, 5 if kind == "batch" else 3)
    elif kind == "voxelize":
        kw["grid"] = _log_int(rng, 24, 512)
        width = height = 16
    elif kind == "voxel_image":
        kw["grid"] = _log_int(rng, 24, 200)
        kw["precision"] = "recheck"
    else:
        kw["frames"] = rng.randint(4, 16)
        width = height = rng.choice([256, 512, 1024])
    c = _case("", kind, width, height, **kw)
    del c["name"]
    return c


def _scenes(case: dict, seed: int) -> list:
    """The case's scenes: sizes by the case alone, constants by the seed."""
    sizes = np.random.default_rng(11)
    out = []
    for i in range(case["frames"]):
        rng = np.random.default_rng([seed, i])
        if case["c"] == "uniform":
            c = scenes.random_c(rng)
        elif case["c"] == "walk":  # a parameter exploration around the default constant
            c = (np.array(scenes.C_DEFAULT) + rng.normal(0.0, 0.02, 8)).tolist()
        else:  # a constant of the paper's captions, moved a little
            names = sorted(scenes.PAPER_C_VALUES)
            c = (np.array(scenes.PAPER_C_VALUES[names[int(rng.integers(len(names)))]])
                 + rng.normal(0.0, 0.005, 8)).tolist()
        w, h, mi = case["width"], case["height"], case["max_iter"]
        if case["kind"] == "served":  # sizes up to the case's, weighted as the serving stream's
            res = [r for r in scenes.RESOLUTIONS if r[0] <= w and r[1] <= h]
            p = np.array(scenes.SERVE_RES_WEIGHTS[:len(res)])
            w, h = res[int(sizes.choice(len(res), p=p / p.sum()))]
            mi = int(sizes.integers(8, 33))
        s = scenes.default_scene(c=c, width=w, height=h, max_iter=mi, march_steps=case["march_steps"],
                                 bisect_steps=case["bisect_steps"], precision=PRECISION[case["precision"]],
                                 traversal=TRAVERSAL[case["traversal"]], modulus_mode=case["modulus"],
                                 square_mode=case["square"])
        if case["slice"] == "random":
            s["slice_basis"] = scenes.random_slice_frame(rng)
        if case["kind"] == "voxel_image":  # an off-axis view, as a user turns the grid
            s["eye"] = (np.array([0.37, 0.23, 3.4]) + rng.normal(0.0, 0.02, 3)).tolist()
            s["target"] = [0.05, -0.11, 0.02]
        out.append(s)
    return out


_contexts: dict = {}


def _context(name: str) -> int:
    """The process's library context (a program keeps one; serving runs on its own)."""
    if name not in _contexts:
        _contexts[name] = binding.dqj_create(0)
    return _contexts[name]


def _planes(s: dict, device: str) -> dict:
    o = binding.alloc_outputs(s["width"], s["height"], device=device, stats=False)
    return {k: (v.pin_memory() if device == "cpu" and torch.is_tensor(v) else v) for k, v in o.items()}


def prepare(case: dict, seed: int) -> dict:
    sc = _scenes(case, seed)
    st = {"kind": case["kind"], "scenes": sc, "grid": case["grid"],
          "ctx": _context("serve" if case["kind"] == "served" else "render")}
    if case["kind"] in ("voxelize", "voxel_image"):
        g = case["grid"]
        st["occupancy"] = torch.empty(g ** 3, dtype=torch.uint8, device="cuda")
        if case["kind"] == "voxelize":
            st["counts"] = torch.empty(g ** 3, dtype=torch.int16, device="cuda")
        else:
            binding.dqj_voxelize(st["ctx"], sc[0], g, st["occupancy"],
                                 stream=torch.cuda.current_stream().cuda_stream)
    if case["kind"] != "voxelize":
        st["planes"] = [_planes(s, "cpu" if case["kind"] == "host" else "cuda") for s in sc]
        st["outputs"] = [binding.outputs_of(o) for o in st["planes"]]
    return st


def run(st: dict):
    ctx, sc = st["ctx"], st["scenes"]
    kind = st["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "render":
        binding.dqj_render(ctx, sc[0], st["outputs"][0], stream)
    elif kind == "batch":
        binding.dqj_render_batch(ctx, sc, st["outputs"], stream)
    elif kind == "host":
        binding.dqj_render_host_batch(ctx, sc, st["outputs"])
    elif kind == "voxelize":
        binding.dqj_voxelize(ctx, sc[0], st["grid"], st["occupancy"], st["counts"], stream=stream)
        return {"occupancy": st["occupancy"], "counts": st["counts"]}
    elif kind == "voxel_image":
        binding.dqj_render_voxels(ctx, sc[0], st["grid"], st["occupancy"], st["outputs"][0], stream)
    else:  # served: submit the burst, poll until every request is done
        pending = [binding.dqj_submit(ctx, s, o) for s, o in zip(sc, st["outputs"])]
        while pending:
            left = []
            for t in pending:
                done, status = binding.dqj_poll(ctx, t)
                if done:
                    binding.check(status)
                else:
                    left.append(t)
            pending = left
    return [{k: o[k] for k in PLANES} for o in st["planes"]]


def work(case: dict) -> dict:
    """Bytes: every output plane (24 bytes a pixel, 3 bytes a cell) written once
    and an occupancy grid read once.  Flops: an FMA counts two, one step of the
    iteration with its escape test 52; a traced pixel needs its camera ray
    (about 60) and at least one whole orbit, a cell at least one step, a pixel of
    a grid's image its ray and about 10 for each of g cells crossed."""
    sc = _scenes(case, 0)
    px = float(sum(s["width"] * s["height"] for s in sc))
    g = case["grid"]
    if case["kind"] == "voxelize":
        return {"bytes": 3.0 * g ** 3, "flops": 52.0 * g ** 3}
    if case["kind"] == "voxel_image":
        return {"bytes": 24.0 * px + g ** 3, "flops": (60.0 + 10.0 * g) * px}
    return {"bytes": 24.0 * px,
            "flops": float(sum(s["width"] * s["height"] * (60.0 + 52.0 * s["max_iter"]) for s in sc))}


# ---------------------------------------------------------------------------
# FP64 values in plain torch
# ---------------------------------------------------------------------------
_SAMPLES = 1 << 22  # samples classified at a time


def _rows(v):
    return torch.tensor(v, dtype=torch.float64, device="cuda")


def _rays(s: dict, pix):
    """Camera rays of linear pixels: unit direction [n, 3], box clip t_in, t_out, crosses."""
    eye, target, up = (np.array(s[k], dtype=np.float64) for k in ("eye", "target", "up"))
    f = target - eye
    f /= np.linalg.norm(f)
    r = np.cross(f, up)
    r /= np.linalg.norm(r)
    u = np.cross(r, f)
    w, h = s["width"], s["height"]
    th = np.tan(np.radians(s["fov_y_deg"]) / 2)
    x, y = (pix % w).double(), torch.div(pix, w, rounding_mode="floor").double()
    sx = (2 * (x + 0.5) / w - 1) * th * (w / h)
    sy = (1 - 2 * (y + 0.5) / h) * th
    d = _rows(f)[None] + sx[:, None] * _rows(r)[None] + sy[:, None] * _rows(u)[None]
    d = d / d.norm(dim=1, keepdim=True)
    e, lo, hi = _rows(s["eye"]), _rows(s["box_min"]), _rows(s["box_max"])
    a, b = (lo - e)[None] / d, (hi - e)[None] / d
    flat = d == 0
    within = ((e >= lo) & (e <= hi))[None].expand_as(d)
    near = torch.where(flat, -torch.inf, torch.minimum(a, b)).amax(dim=1).clamp(min=0.0)
    far = torch.where(flat, torch.inf, torch.maximum(a, b)).amin(dim=1)
    return d, near, far, (near < far) & (within | ~flat).all(dim=1)


def _point(s: dict, p):
    """Slice image of scene points [..., 3], as a list of eight components."""
    e, o = np.array(s["slice_basis"]), s["slice_origin"]
    return [o[i] + p[..., 0] * e[0, i] + p[..., 1] * e[1, i] + p[..., 2] * e[2, i] for i in range(8)]


def _step(z, s: dict):
    c = s["c"]

    def sq(q):
        return [q[0] * q[0] - q[1] * q[1] - q[2] * q[2] - q[3] * q[3], 2 * q[0] * q[1], 2 * q[0] * q[2],
                2 * q[0] * q[3]]
    r, d = z[:4], z[4:]
    if s["square_mode"] == 0:
        dd = [2 * (r[0] * d[0] - r[1] * d[1] - r[2] * d[2] - r[3] * d[3])]
        dd += [2 * (r[0] * d[i] + d[0] * r[i]) for i in (1, 2, 3)]
    else:
        dd = sq(d)
    return [v + c[i] for i, v in enumerate(sq(r) + dd)]


def _modulus(z, s: dict):
    n = 8 if s["modulus_mode"] == 0 else 4
    m = z[0] * z[0]
    for v in z[1:n]:
        m = m + v * v
    return m


def _classify(z, s: dict, estimate=False):
    """Escape count of flat samples (0: inside), and the distance estimate."""
    n = torch.zeros(z[0].shape, dtype=torch.int32, device="cuda")
    dist = torch.zeros_like(z[0])
    live = torch.arange(z[0].numel(), device="cuda")
    r2 = s["escape_radius"] ** 2
    m = _modulus(z, s) if estimate else None
    dr2 = torch.ones_like(z[0])
    for it in range(1, s["max_iter"] + 1):
        if estimate:
            dr2 = 4 * m * dr2
        z = _step(z, s)
        m = _modulus(z, s)
        out = m > r2
        n[live[out]] = it
        if estimate:
            dist[live[out]] = 0.25 * torch.sqrt(m[out] / dr2[out]) * torch.log(m[out])
        keep = ~out
        z = [v[keep] for v in z]
        live, m, dr2 = live[keep], m[keep], dr2[keep]
        if live.numel() == 0:
            break
    return n, dist


def _normal(s: dict, p, d, n):
    """Central differences of the modulus after n steps at points p; -d where it vanishes or overflows."""
    f = []
    for a in range(3):
        for sign in (1.0, -1.0):
            q = p.clone()
            q[:, a] += sign * s["normal_h"]
            z = _point(s, q)
            for it in range(int(n.max()) if n.numel() else 0):
                w = _step(z, s)
                z = [torch.where(n > it, x, y) for x, y in zip(w, z)]
            f.append(_modulus(z, s))
    f = torch.stack(f, dim=1)
    g = f[:, 0::2] - f[:, 1::2]
    big = g.abs().amax(dim=1, keepdim=True)
    bad = ~(f <= 2.0 ** 100).all(dim=1) | ~(big[:, 0] > 0)
    g = g / big
    g = g / g.norm(dim=1, keepdim=True)
    return torch.where(bad[:, None], -d, g)


def _march(s: dict, pix):
    d, t0, t1, ok = _rays(s, pix)
    depth = torch.full((pix.numel(),), torch.inf, dtype=torch.float64, device="cuda")
    normal = torch.zeros((pix.numel(), 3), dtype=torch.float64, device="cuda")
    sel = ok.nonzero()[:, 0]
    if sel.numel() == 0:
        return depth, normal
    d, t0, t1 = d[sel], t0[sel], t1[sel]
    steps = s["march_steps"]
    delta = (t1 - t0) / steps
    k = torch.arange(steps + 1, device="cuda", dtype=torch.float64)
    t = t0[:, None] + k[None] * delta[:, None]
    eye = _rows(s["eye"])
    p = eye + t[..., None] * d[:, None, :]
    n = _classify([v.reshape(-1) for v in _point(s, p)], s)[0].reshape(t.shape)
    inside = n == 0
    hit = inside.any(dim=1)
    first = inside.int().argmax(dim=1)
    sel, d, t0, delta, first, n = sel[hit], d[hit], t0[hit], delta[hit], first[hit], n[hit]
    if sel.numel() == 0:
        return depth, normal
    prev = n.gather(1, (first - 1).clamp(min=0)[:, None].long())[:, 0]
    start = first == 0
    star = torch.where(start, torch.full_like(prev, s["max_iter"]), prev)
    lo, hi = t0 + (first - 1).double() * delta, t0 + first.double() * delta
    for _ in range(s["bisect_steps"]):
        mid = lo + 0.5 * (hi - lo)
        m = _classify(_point(s, eye + mid[:, None] * d), s)[0]
        star = torch.where((m > 0) & ~start, m, star)
        lo, hi = torch.where(m > 0, mid, lo), torch.where(m > 0, hi, mid)
    at = torch.where(start, t0, lo + 0.5 * (hi - lo))
    depth[sel] = at
    normal[sel] = _normal(s, eye + at[:, None] * d, d, star)
    return depth, normal


def _sphere_trace(s: dict, pix):
    d, t0, t1, ok = _rays(s, pix)
    depth = torch.full((pix.numel(),), torch.inf, dtype=torch.float64, device="cuda")
    star = torch.zeros(pix.numel(), dtype=torch.int32, device="cuda")
    live = ok.nonzero()[:, 0]
    t = t0.clone()
    eye = _rows(s["eye"])
    for _ in range(s["de_max_steps"]):
        if live.numel() == 0:
            break
        n, dist = _classify(_point(s, eye + t[live][:, None] * d[live]), s, estimate=True)
        stop = (n == 0) | (dist < s["de_epsilon"])
        at = live[stop]
        depth[at] = t[at]
        star[at] = torch.where(n[stop] > 0, n[stop], torch.full_like(n[stop], s["max_iter"]))
        live, dist = live[~stop], dist[~stop]
        t[live] += s["de_step_scale"] * dist
        live = live[t[live] <= t1[live]]
    hit = torch.isfinite(depth)
    normal = torch.zeros((pix.numel(), 3), dtype=torch.float64, device="cuda")
    if hit.any():
        normal[hit] = _normal(s, eye + depth[hit][:, None] * d[hit], d[hit], star[hit])
    return depth, normal


def _grid_image(s: dict, g: int, pix):
    e, lo, hi = _rows(s["eye"]), _rows(s["box_min"]), _rows(s["box_max"])
    size = (hi - lo) / g
    occ = []
    for k in range(g):  # occupancy by cell centres, one z slice at a time
        i = (torch.arange(g, device="cuda", dtype=torch.float64) + 0.5)
        y, x = torch.meshgrid(lo[1] + i * size[1], lo[0] + i * size[0], indexing="ij")
        c = torch.stack([x, y, torch.full_like(x, float(lo[2] + (k + 0.5) * size[2]))], dim=-1).reshape(-1, 3)
        occ.append(_classify(_point(s, c), s)[0] == 0)
    occ = torch.cat(occ)
    d, t0, t1, ok = _rays(s, pix)
    depth = torch.full((pix.numel(),), torch.inf, dtype=torch.float64, device="cuda")
    normal = torch.zeros((pix.numel(), 3), dtype=torch.float64, device="cuda")
    near = torch.minimum((lo - e) / d, (hi - e) / d)
    face = torch.where(near.amax(dim=1) > 0, near.argmax(dim=1), torch.full_like(pix, -1))
    live = ok.nonzero()[:, 0]
    step = torch.sign(d).long()
    cell = ((e + t0[:, None] * d - lo) / size).floor().clamp(0, g - 1).long()
    entry = t0.clone()
    for _ in range(3 * g):
        if live.numel() == 0:
            break
        c = cell[live]
        found = occ[(c[:, 2] * g + c[:, 1]) * g + c[:, 0]]
        at = live[found]
        depth[at] = entry[at]
        ax = face[at]
        n = torch.zeros((at.numel(), 3), dtype=torch.float64, device="cuda")
        n.scatter_(1, ax.clamp(min=0)[:, None], -torch.sign(d[at]).gather(1, ax.clamp(min=0)[:, None]))
        normal[at] = torch.where(ax[:, None] < 0, -d[at], n)
        live = live[~found]
        c, dl = cell[live], d[live]
        plane = c + (step[live] > 0).long()
        dist = torch.where(dl == 0, torch.inf, (lo + plane * size - e) / dl)
        a = dist.argmin(dim=1)
        face[live] = a
        entry[live] = dist.gather(1, a[:, None])[:, 0]
        c = c.scatter_add(1, a[:, None], step[live].gather(1, a[:, None]))
        cell[live] = c
        live = live[((c >= 0) & (c < g)).all(dim=1)]
    return depth, normal


def exact(case: dict, seed: int):
    """Depth and normal planes in FP64; the others are whole numbers."""
    if case["kind"] == "voxelize":
        return None
    out = []
    for s in _scenes(case, seed):
        n = s["width"] * s["height"]
        if case["kind"] == "voxel_image" or case["traversal"] == "de":
            size = n
        else:
            size = max(1, _SAMPLES // (s["march_steps"] + 1))
        depth, normal = [], []
        for a in range(0, n, size):
            pix = torch.arange(a, min(n, a + size), device="cuda")
            if case["kind"] == "voxel_image":
                v = _grid_image(s, case["grid"], pix)
            else:
                v = _sphere_trace(s, pix) if case["traversal"] == "de" else _march(s, pix)
            depth.append(v[0])
            normal.append(v[1])
        shape = (s["height"], s["width"])
        depth, normal = torch.cat(depth).reshape(shape), torch.cat(normal).reshape(shape + (3,))
        if case["kind"] == "host":
            depth, normal = depth.cpu(), normal.cpu()
        out.append({"iter": None, "depth": depth, "normal": normal, "rgba": None})
    return out
