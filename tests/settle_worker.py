"""Renders the settled-block scenes and saves every plane and counter (run by
tests/test_gpu_settle.py under DQJ_MARCH_SAMPLES = 0 and 2)."""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from paper_2303_14827_gb300 import binding, scenes  # noqa: E402


def scene_list():
    """Sample counts at the edges of pairs, blocks and chunks; every precision,
    square and modulus; axis, rotated-axis and random slices; eyes inside,
    grazing and far from the box; escape radii, margins, iteration limits and
    boxes at the ends of what is in use."""
    out = []

    def add(**kw):
        frame = kw.pop("frame", None)
        s = scenes.default_scene(**dict(dict(width=77, height=45, bisect_steps=4), **kw))
        if frame is not None:
            s["slice_basis"] = frame
        out.append(s)

    rng = np.random.default_rng(31)
    slice8 = scenes.random_slice_frame(rng)
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    axis3 = np.zeros((3, 8))
    axis3[:, :3] = q
    frames = (None, slice8, axis3.tolist())
    for i, n in enumerate((1, 2, 7, 8, 9, 15, 16, 62, 63, 64, 65, 127, 255, 509, 510, 511, 512, 513, 700, 1023, 1025)):
        for prec in (0, 1, 2):
            add(march_steps=n, precision=prec, frame=frames[i % 3], c=scenes.random_c(rng) if i % 2 else
                list(scenes.C_DEFAULT), max_iter=12 + i)
    for prec in (0, 1, 2):
        for sq in (0, 1):
            for mod in (0, 1):
                add(precision=prec, square_mode=sq, modulus_mode=mod, frame=frames[sq + mod], max_iter=24)
        for kw in (dict(max_iter=1), dict(max_iter=2), dict(max_iter=3, frame=slice8), dict(escape_radius=0.7),
                   dict(escape_radius=50.0, frame=slice8), dict(recheck_margin=0.0), dict(recheck_margin=0.5),
                   dict(c=[0.0] * 8), dict(c=[3.0, 0, 0, 0, 2.0, 0, 0, 0]), dict(c=[1e20, 0, 0, 0, 0, 0, 0, 1e20]),
                   dict(eye=[0.1, 0.2, 0.3], target=[1.0, 0.4, 0.2]), dict(eye=[1.99, 0.0, 1.99]),
                   dict(eye=[300.0, 20.0, 350.0], fov_y_deg=1.0), dict(eye=[2.6, 2.4, 2.7], fov_y_deg=100.0),
                   dict(box_min=[-50.0] * 3, box_max=[50.0] * 3), dict(box_min=[-0.1, -2, -1], box_max=[0.4, 0.1, 1.7]),
                   dict(box_min=[-1e12] * 3, box_max=[1e12] * 3), dict(width=1, height=1), dict(width=640, height=9),
                   dict(slice_origin=[0, 0, 0, 0.3, 0.1, -0.2, 0.4, 0.0])):
            add(precision=prec, march_steps=300, **kw)
    add(width=1280, height=720, march_steps=512, precision=1)  # more tiles than resident warps
    add(width=1280, height=720, march_steps=512, precision=0, frame=slice8, c=scenes.random_c(rng))
    return out


def main(path):
    import torch
    out = {}
    with binding.Renderer(0) as r:
        for i, s in enumerate(scene_list()):
            o = r.render(s)
            for k in ("iter", "depth", "normal", "rgba", "stats"):
                out[f"{i}_{k}"] = o[k].cpu().numpy()
        # voxel grids: edges of bricks and sub-bricks, rows with and without wide stores
        rng = np.random.default_rng(32)
        for i, g in enumerate((64, 71, 100, 336, 337, 345, 352)):
            for prec in (0, 1, 2) if g <= 100 else (0, 1):
                s = scenes.default_scene(precision=prec, max_iter=14, c=scenes.random_c(rng))
                if i % 2:
                    s["slice_basis"] = scenes.random_slice_frame(rng)
                occ = torch.full((g ** 3,), 7, dtype=torch.uint8, device="cuda")
                cnt = torch.full((g ** 3,), 7, dtype=torch.int16, device="cuda")
                st = torch.zeros(binding.DQJ_NSTATS, dtype=torch.int64, device="cuda")
                binding.dqj_voxelize(r.ctx, s, g, occ, cnt, st, torch.cuda.current_stream().cuda_stream)
                tag = f"voxel{g}p{prec}"
                planes = torch.arange(g ** 3, device="cuda") % 8191 + 1  # weights: a grid as a few sums
                out[tag + "_iter"] = np.array([int(occ.sum()), int((occ.long() * planes).sum())])
                out[tag + "_count"] = np.array([int(cnt.sum()), int((cnt.long() * planes).sum())])
                st[4:7] = 0  # how many cells were rechecked depends on the cells that share a warp's steps
                out[tag + "_stats"] = st.cpu().numpy()
        torch.cuda.synchronize()
    np.savez(path, **out)


if __name__ == "__main__":
    main(sys.argv[1])
