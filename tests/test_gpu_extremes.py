"""Calls at the ends of what the parameters allow: boxes whose samples overflow."""
import numpy as np
import pytest

from paper_2303_14827_gb300 import binding, scenes
from parity import to_numpy

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
