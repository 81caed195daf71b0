"""Calls at the ends of what the parameters allow: boxes whose samples overflow,
escape radii below what FP32 squares resolve, rays that run almost parallel
to a slab they lie outside of, and eyes beside the box's faces and corners."""
import numpy as np
import pytest

import oracle
from paper_2303_14827_gb300 import binding, scenes
from parity import assert_parity, compare, to_numpy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("general", (False, True))
@pytest.mark.parametrize("square,modulus", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("precision,half", [(2, 1e160), (2, 1e200), (1, 1e25), (0, 1e25)])
def test_overflowing_samples_escape(square, modulus, precision, half, general):
    # the halves of such a sample's square are differences of infinities: neither
    # bounded nor inside
    import torch
    s = scenes.default_scene(width=40, height=24, march_steps=20, precision=precision, square_mode=square,
                             modulus_mode=modulus, box_min=[-half] * 3, box_max=[half] * 3,
                             eye=[-7.0, 5.0, 6.0], target=[-8.0, 6.1, 7.3])
    if general:
        s["slice_basis"] = scenes.random_slice_frame(np.random.default_rng(3))
    with binding.Renderer(0) as r:
        g = to_numpy(r.render(s), 40, 24)
        assert np.all(np.isinf(g["depth"])) and np.all(g["iter"] == 1)
        n = 10
        occ = torch.full((n ** 3,), 7, dtype=torch.uint8, device="cuda")
        cnt = torch.full((n ** 3,), 7, dtype=torch.int16, device="cuda")
        binding.dqj_voxelize(r.ctx, s, n, occ, cnt, None, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert not occ.any() and bool((cnt == 1).all())


@pytest.mark.parametrize("radius", (1e-22, 1e-19, 1e-16, 1e-11))
def test_fp64_tiny_radius(radius):
    # |zeta_1|^2 against R^2 = 1e-44 .. 1e-22: subnormal or nearly so in FP32
    u = radius ** 0.5
    c = [0.3 * radius, -0.2 * radius, 0.1 * radius, 0.0, 0.1 * radius, 0.0, 0.0, 0.05 * radius]
    s = scenes.default_scene(width=72, height=40, precision=2, escape_radius=radius, c=c, normal_h=1e-4 * u,
                             box_min=[-2 * u] * 3, box_max=[2 * u] * 3, eye=[0.4 * u, 0.3 * u, 3.5 * u],
                             target=[0.0, 0.1 * u, 0.0])
    with binding.Renderer(0) as r:
        g = to_numpy(r.render(s), 72, 40)
    o = oracle.render(s)
    hg, ho = np.isfinite(g["depth"]), np.isfinite(o["depth"])
    assert 100 < ho.sum() < 2800
    assert np.array_equal(hg, ho) and np.array_equal(g["iter"], o["iter"])
    # a bracket is 3 u / 256 / 2^8 long; a decision within FP64 rounding moves it by one last place
    assert np.abs(g["depth"][ho].astype(np.float64) - o["depth"][ho]).max() <= 1e-6 * 4 * u


@pytest.mark.parametrize("g", (8, 24, 100))
@pytest.mark.parametrize("side", (1.0, -1.0))
def test_voxel_ray_beside_the_grid(g, side):
    # direction 2e-41 along y, the eye outside the box on y: no ray meets the grid
    import torch
    s = scenes.default_scene(width=64, height=1, eye=[5.0, 1e-40, 0.0], target=[0.0, 0.0, 0.0],
                             box_min=[-2.0, -2.0 if side > 0 else 1.0, -2.0],
                             box_max=[2.0, -1.0 if side > 0 else 2.0, 2.0])
    occ = np.ones((g, g, g), dtype=np.uint8)
    assert not np.isfinite(oracle.voxel_render(s, occ)["depth"]).any()
    with binding.Renderer(0) as r:
        t = binding.alloc_outputs(64, 1, stats=False)
        d_occ = torch.from_numpy(occ.reshape(-1)).cuda()
        binding.dqj_render_voxels(r.ctx, s, g, d_occ, binding.outputs_of(t), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        out = to_numpy(t, 64, 1)
    assert np.all(np.isinf(out["depth"])) and np.all(out["iter"] == 0)


@pytest.mark.parametrize("precision", (1, 2))
@pytest.mark.parametrize("off", (1e-3, 1e-4, 1e-6, -1e-3, -1e-6))
@pytest.mark.parametrize("sides", [(1, 1, 1.3), (0, 1, 0), (1, 0, 1.7), (-1, -1, -1)])
def test_eye_beside_the_box(sides, off, precision):
    # off > 0 outside, < 0 inside; 0 in sides: well inside the slab
    eye = [2.0 * np.sign(d) + off * d if d else 0.31 for d in sides]
    s = scenes.default_scene(width=96, height=72, precision=precision, eye=eye, target=[0.05, -0.11, 0.02],
                             fov_y_deg=60.0, march_steps=400, bisect_steps=8, max_iter=16)
    with binding.Renderer(0) as r:
        g = to_numpy(r.render(s), 96, 72)
    assert_parity(compare(g, oracle.render(s)), what=f"eye {eye}")
