"""Renders frames that settle blocks and decide samples by bounds, and saves every
plane and counter (run by tests/test_gpu_decisions.py with and without the
bounds: DQJ_BOUNDS, DQJ_MARCH_SAMPLES)."""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from paper_2303_14827_gb300 import binding, scenes  # noqa: E402


def scene_list():
    """Narrow views, whose tiles are thin enough for the march to settle blocks:
    odd and even sample counts at the edges of blocks and chunks, both squares and
    moduli, axis, rotated-axis and random slices, FP32, recheck and FP64; then
    whole frames at the sizes in use.  Bisection steps, iteration limits and margins keep the
    recheck queue (four entries a pixel) from overflowing where every pixel is a
    hit, or where every bounded orbit is a late one."""
    out = []
    rng = np.random.default_rng(41)
    slice8 = scenes.random_slice_frame(rng)
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    axis3 = np.zeros((3, 8))
    axis3[:, :3] = q
    frames = (None, slice8, axis3.tolist())

    def add(**kw):
        frame = kw.pop("frame", None)
        s = scenes.default_scene(**dict(dict(width=77, height=45, fov_y_deg=3.0, eye=[0.3, 0.2, 3.5],
                                             target=[0.25, 0.75, 0.0], bisect_steps=2, max_iter=20), **kw))
        if frame is not None:
            s["slice_basis"] = frame
        out.append(s)

    for i, n in enumerate((190, 255, 256, 257, 319, 320, 321, 448, 509, 510, 511, 512, 513, 700, 1023, 1024, 1025, 1537)):
        for prec in (0, 1):
            add(march_steps=n, precision=prec, frame=frames[i % 3], max_iter=8 + i % 13, recheck_margin=1e-4)
    for prec in (0, 1, 2):
        for sq in (0, 1):
            for mod in (0, 1):
                for f in frames:
                    add(march_steps=400, precision=prec, square_mode=sq, modulus_mode=mod, frame=f,
                        target=[0.1, 0.6, 0.0], fov_y_deg=4.0,
                        max_iter=30 if prec != 1 else 12 if mod else 20, recheck_margin=2e-4)
    wide = dict(fov_y_deg=45.0, eye=[0.1, 0.2, 3.5], target=[0.0, 0.0, 0.0], march_steps=512)
    for sq in (0, 1):
        for mod in (0, 1):
            for prec in (1, 2):
                for f in (None, slice8):
                    w, h = (481, 271) if prec == 2 else (640, 400)
                    add(**dict(wide, width=w, height=h, precision=prec, square_mode=sq, modulus_mode=mod, frame=f,
                               max_iter=22 + 4 * sq + 2 * mod, bisect_steps=2 if prec == 1 else 10,
                               c=(np.array(scenes.C_DEFAULT) + rng.normal(0, 0.02, 8)).tolist()))
    for c in (scenes.C_DEFAULT, scenes.random_c(rng)):
        add(**dict(wide, width=1920, height=1080, precision=1, c=list(c), max_iter=16,
                   bisect_steps=10))
    return out


def main(path):
    import torch
    out = {}
    with binding.Renderer(0) as r:
        for i, s in enumerate(scene_list()):
            o = r.render(s)
            for k in ("iter", "depth", "normal", "rgba", "stats"):
                out[f"{i}_{k}"] = o[k].cpu().numpy()
        rng = np.random.default_rng(42)
        for g in (64, 337, 400):
            for prec in (0, 1, 2) if g < 400 else (1,):
                for sq in (0, 1):
                    s = scenes.default_scene(precision=prec, max_iter=20, c=scenes.random_c(rng), square_mode=sq,
                                             modulus_mode=(g + prec) % 2)
                    occ = torch.empty(g ** 3, dtype=torch.uint8, device="cuda")
                    cnt = torch.empty(g ** 3, dtype=torch.int16, device="cuda")
                    binding.dqj_voxelize(r.ctx, s, g, occ, cnt, None, torch.cuda.current_stream().cuda_stream)
                    at = torch.arange(g ** 3, device="cuda") % 8191 + 1  # weights: a grid as a few sums
                    out[f"voxel{g}p{prec}s{sq}_iter"] = np.array(
                        [int(occ.sum()), int((occ.long() * at).sum()), int(cnt.sum()), int((cnt.long() * at).sum())])
        torch.cuda.synchronize()
    np.savez(path, **out)


if __name__ == "__main__":
    main(sys.argv[1])
