"""The recheck's device functions against plain FP64, called one by one through a
probe library built from the same headers (bounds_probe.cu): the FP64 clip of a
ray, the positions of samples, the two orbit bounds, the bound of a march
sample's position, the FP64 doublings on the integer units, and what becomes of
staged samples that find the recheck queue full."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2303_14827_gb300 import binding, build, scenes

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
I32, U64 = ctypes.POINTER(ctypes.c_int32), ctypes.POINTER(ctypes.c_uint64)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    binding.load()
    so = str(tmp_path_factory.mktemp("probe") / "bounds_probe.so")
    cmd = [build._nvcc(), "-shared", "-Xcompiler", "-fPIC", "-std=c++17", "-O3"] + build.ARCH + [
        "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC, os.path.join(HERE, "bounds_probe.cu"),
        "-o", so, "-cudart", "shared", "-L", build.HERE, "-l:libdqj.so", "-Xlinker", "-rpath," + build.HERE]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return ctypes.CDLL(so)


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def scene_params(**kw):
    return binding.make_params(scenes.default_scene(**kw))


BOXES = (([-2.0] * 3, [2.0] * 3), ([-2.1, -1.7, -0.3], [1.9, 2.3, 1.1]))


@pytest.mark.parametrize("off", (1e-3, 1e-4, 1e-5, 1e-6, 1e-8, 0.5))
@pytest.mark.parametrize("box", range(len(BOXES)))
def test_ray_clip(probe, off, box):
    # eyes beside a face, an edge and a corner, outside and inside: face - eye
    # cancels.  Exact to the rounding of the difference, the reciprocal and the
    # product: 3 units of 2^-53, 8 allowed.
    import torch
    lo, hi = np.array(BOXES[box][0]), np.array(BOXES[box][1])
    w, h = 96, 80
    xs, ys = np.meshgrid(np.arange(w, dtype=np.int32), np.arange(h, dtype=np.int32))
    dx, dy = dev(xs.ravel()), dev(ys.ravel())
    mid = 0.5 * (lo + hi)
    tested = 0
    for sides in ((1, 1, 1.3), (1, 1, 0), (0, 1.1, 1), (0, 0, 1), (-1, 1.7, 1), (-1, -1, -1), (-1, 0, 0), (1, -1.2, 0.01)):
        for corner in (hi, lo):
            out = np.where(corner == hi, 1.0, -1.0)
            eye = np.where(np.array(sides) == 0, mid + 0.21, corner + out * off * np.array(sides))
            p = scene_params(width=w, height=h, eye=eye.tolist(), target=(mid + [0.07, -0.13, 0.11]).tolist(),
                             box_min=lo.tolist(), box_max=hi.tolist(), fov_y_deg=80.0)
            t = torch.empty(2, w * h, dtype=torch.float64, device="cuda")
            ray = torch.empty(w * h, 3, dtype=torch.float64, device="cuda")
            assert probe.probe_clip(ctypes.byref(p), ptr(dx), ptr(dy), w * h, ptr(t[0]), ptr(t[1]), ptr(ray)) == 0
            d = ray.cpu().numpy().astype(np.longdouble)
            e = eye.astype(np.longdouble)
            with np.errstate(all="ignore"):
                a, b = (lo - e) / d, (hi - e) / d
            t0 = np.maximum(np.minimum(a, b).max(1), 0)
            t1 = np.maximum(a, b).min(1)
            ok = np.isfinite(t0) & np.isfinite(t1) & (t0 < t1)
            tested += int(ok.sum())
            got = t.cpu().numpy()
            for g, want in ((got[0], t0), (got[1], t1)):
                err = np.abs(g - want)[ok]
                bad = err > 8 * 2.0 ** -53 * np.abs(want[ok])
                assert not bad.any(), (sides, int(bad.sum()), float(err.max()))
    assert tested > 20000


def ray_points(s, cam, x, y, k, T):
    """Slice points of march samples by the reference formula in type T, from the
    library's own (FP64) camera constants, and which of the rays cross the box."""
    t = {n: np.array(s[n], dtype=T) for n in ("eye", "box_min", "box_max", "slice_origin", "slice_basis")}
    f, r, u = (cam[3 * a:3 * a + 3].astype(T) for a in range(3))
    th, aspect = T(cam[9]), T(cam[10])
    sx = (2 * (x.astype(T) + T(0.5)) / s["width"] - 1) * th * aspect
    sy = (1 - 2 * (y.astype(T) + T(0.5)) / s["height"]) * th
    d = f + sx[:, None] * r + sy[:, None] * u
    d = d / np.sqrt((d * d).sum(1))[:, None]
    with np.errstate(all="ignore"):
        a, b = (t["box_min"] - t["eye"]) / d, (t["box_max"] - t["eye"]) / d
    t0 = np.maximum(np.fmin(a, b).max(1), 0)
    t1 = np.fmax(a, b).min(1)
    tau = t0 + k.astype(T) * ((t1 - t0) / s["march_steps"])
    return t["slice_origin"] + (t["eye"] + tau[:, None] * d) @ t["slice_basis"], t1 - t0 > 1e-3


@pytest.mark.parametrize("eye", ([0.37, 0.23, 3.4], [2.3, 1.1, 2.6], [0.1, 0.2, 0.3]))
@pytest.mark.parametrize("seed", (None, 1, 2))
def test_sample_positions(probe, eye, seed):
    # the recheck places its samples as closely as the reference formula in FP64
    # does (rms over many samples; the two differ by sampling, a few per cent)
    import torch
    assert np.finfo(np.longdouble).nmant >= 63
    rng = np.random.default_rng(23)
    n = 60000
    s = scenes.default_scene(width=1920, height=1080, march_steps=512, precision=1, eye=eye, target=[0.05, -0.11, 0.02])
    if seed is not None:
        s["slice_basis"] = scenes.random_slice_frame(np.random.default_rng(seed))
    x, y, k = (rng.integers(0, m, n).astype(np.int32) for m in (1920, 1080, 513))
    p = binding.make_params(s)
    cam = np.empty(11)
    probe.probe_camera(ctypes.byref(p), ctypes.c_void_p(cam.ctypes.data))
    exact, ok = ray_points(s, cam, x, y, k, np.longdouble)
    plain, _ = ray_points(s, cam, x, y, k, np.float64)
    z = torch.empty(n, 8, dtype=torch.float64, device="cuda")
    dx, dy, dk = dev(x), dev(y), dev(k)
    assert probe.probe_positions(ctypes.byref(p), ptr(dx), ptr(dy), ptr(dk), n, ptr(z)) == 0

    def rms(v):
        return float(np.sqrt((((v - exact)[ok]) ** 2).sum(1).mean()))

    assert ok.sum() > n // 8
    assert rms(z.cpu().numpy()) <= 1.05 * rms(plain)


def classify(probe, p, which, z):
    import torch
    zd = dev(z)
    out = torch.empty(2, len(z), dtype=torch.int32, device="cuda")
    assert probe.probe_count(ctypes.byref(p), which, ptr(zd), len(z), ptr(out[0]), ptr(out[1])) == 0
    return out.cpu().numpy()


@pytest.mark.parametrize("square", (0, 1))
@pytest.mark.parametrize("modulus", (0, 1))
@pytest.mark.parametrize("radius", (0.7, 4.0, 50.0))
def test_orbit_bounds(probe, square, modulus, radius):
    # random points, and points where the FP64 count changes (bisected down to
    # neighbouring doubles), axis slices and general ones: a certain count is the
    # FP64 evaluation's, and count64 always is
    rng = np.random.default_rng(7)
    n = 4000
    decided = [0, 0]
    for axis in (True, False):
        for c in (list(scenes.C_DEFAULT), scenes.random_c(rng), [0.0] * 8, [0.25] + [0.0] * 7):
            kw = dict(c=c, square_mode=square, modulus_mode=modulus, escape_radius=radius, max_iter=32)
            if not axis:
                kw["slice_basis"] = scenes.random_slice_frame(rng)
            p = scene_params(**kw)
            z = rng.uniform(-1.6, 1.6, (2, n, 8))
            if axis:
                z[..., 3:] = 0.0
            lo, hi = z
            n_lo, n_hi = classify(probe, p, 2, lo)[0], classify(probe, p, 2, hi)[0]
            for _ in range(60):  # lo and hi stay on either side of a change of the count
                m = 0.5 * (lo + hi)
                nm = classify(probe, p, 2, m)[0]
                same = (nm == n_lo)[:, None]
                lo, hi = np.where(same, m, lo), np.where(same, hi, m)
            pts = np.concatenate([z[0], z[1], lo, hi, lo + 1e-9 * (hi - lo) + rng.normal(0, 1e-7, (n, 8)) * (z[0] != 0),
                                  lo + rng.normal(0, 1e-12, (n, 8)) * (z[0] != 0)])
            want = classify(probe, p, 2, pts)[0]
            for which in (0, 1):
                got, certain = classify(probe, p, which, pts)
                bad = (certain != 0) & (got != want)
                assert not bad.any(), (which, axis, c, pts[bad][:2], got[bad][:4], want[bad][:4])
                decided[which] += int(certain.sum())
            assert np.array_equal(classify(probe, p, 3, pts)[0], want)
    assert decided[0] > 0.2 * 48 * n and decided[1] > decided[0]  # the bounds decide something


def test_integer_doubling(probe):
    # every exponent and sign: zeros, subnormals (whose carry enters the exponent),
    # normals, overflow, infinities and NaN
    import torch
    edges = np.array([0, 1, 2, 0x80000000, 0xffffffff, 1 << 32, (1 << 51) - 1, 1 << 51, (1 << 52) - 1], dtype=np.uint64)
    m = np.concatenate([edges, np.random.default_rng(5).integers(0, 1 << 52, 500, dtype=np.uint64)])
    bits = ((np.arange(4096, dtype=np.uint64) << np.uint64(52))[:, None] | m[None]).ravel()
    x = dev(bits.view(np.float64))
    out = torch.empty(2, x.numel(), dtype=torch.float64, device="cuda")
    assert probe.probe_twice(ptr(x), ctypes.c_long(x.numel()), ptr(out[0]), ptr(out[1])) == 0
    with np.errstate(all="ignore"):
        want = bits.view(np.float64) * 2.0, bits.view(np.float64) * 4.0
    for got, w in zip(out.cpu().numpy(), want):
        nan = np.isnan(w)
        assert np.array_equal(np.isnan(got), nan)
        assert np.array_equal(got[~nan].view(np.uint64), w[~nan].view(np.uint64))


VIEWS = (dict(), dict(eye=[2.0001, 2.0001, 2.00013]), dict(eye=[0.3, 1.999, 0.2]), dict(eye=[1.1, 0.4, 0.9]),
         dict(eye=[40.0, 31.0, 55.0], fov_y_deg=4.0), dict(eye=[2.0 + 1e-6, 0.3, 1.0], target=[-1.0, 0.1, 0.2]))


@pytest.mark.parametrize("square", (0, 1))
@pytest.mark.parametrize("modulus", (0, 1))
def test_sample_certain(probe, square, modulus):
    # the FP32 march's count of a sample is certain only where FP64 evaluation
    # from the FP64 position gives the same
    import torch
    rng = np.random.default_rng(11)
    n, w, h, steps = 200000, 640, 360, 512
    right = 0
    for axis in (True, False):
        for view in VIEWS:
            kw = dict(view, c=scenes.random_c(rng), width=w, height=h, march_steps=steps, max_iter=20,
                      square_mode=square, modulus_mode=modulus, precision=1)
            if not axis:
                kw["slice_basis"] = scenes.random_slice_frame(rng)
            s = scenes.default_scene(**kw)
            p = binding.make_params(s)
            with binding.Renderer(0) as r:  # pixels whose rays cross the box
                it = r.render(dict(s, precision=2, march_steps=8))["iter"].cpu().numpy()
            py, px = np.nonzero(it > 0)
            pick = rng.integers(0, len(px), n)
            x, y = px[pick].astype(np.int32), py[pick].astype(np.int32)
            k = rng.integers(0, steps + 1, n).astype(np.int32)
            out = torch.empty(3, n, dtype=torch.int32, device="cuda")
            dx, dy, dk = dev(x), dev(y), dev(k)
            assert probe.probe_samples(ctypes.byref(p), ptr(dx), ptr(dy), ptr(dk), n, ptr(out[0]), ptr(out[1]),
                                       ptr(out[2])) == 0
            o = out.cpu().numpy()
            assert not o[2].any(), (axis, view, int(o[2].sum()))
            right += int(o[1].sum())
    assert right > n  # and it vouches for many of the right ones


@pytest.mark.parametrize("n", (1, 31, 32, 33, 64, 320))
@pytest.mark.parametrize("cap", (0, 1, 40, 1000))
def test_full_queue(probe, n, cap):
    # every staged sample left over is in the queue, or counted as an overflow
    # and its pixel listed for the FP64 re-render
    import torch
    w, h = 64, 45
    p = scene_params(width=w, height=h, precision=1, march_steps=512)
    px = np.arange(n, dtype=np.int32) * 7
    e = np.stack([px, (100 + 0 * px) | (31 << 16), px % w | (px // w << 16), 0 * px + 99], 1).astype(np.int32)
    entries = dev(e)
    queue = torch.zeros(max(cap, 1), 4, dtype=torch.int32, device="cuda")
    flags = torch.zeros(w * h, dtype=torch.int32, device="cuda")
    listed = torch.full((w * h,), -1, dtype=torch.int32, device="cuda")
    oq, od = ctypes.c_int32(), ctypes.c_int32()
    size = probe.probe_counter_offsets(ctypes.byref(oq), ctypes.byref(od))
    ctr = torch.zeros(size, dtype=torch.uint8, device="cuda")
    assert probe.probe_staged(ctypes.byref(p), ptr(entries), n, ptr(queue), cap, ptr(flags), ptr(listed), ptr(ctr)) == 0
    raw = ctr.cpu().numpy()
    stats = raw[:80].view(np.int64)
    queued = min(cap, n)
    assert stats[4] == n
    assert raw[oq.value:oq.value + 4].view(np.uint32)[0] == n
    assert stats[7] == n - queued
    dirty = int(raw[od.value:od.value + 4].view(np.uint32)[0])
    q = queue.cpu().numpy()[:queued, 0]
    d = listed.cpu().numpy()[:dirty]
    assert dirty == n - queued and sorted(np.concatenate([q, d]).tolist()) == px.tolist()
