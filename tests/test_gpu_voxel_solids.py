"""The grid image by blocks of cells on solids, surfaces, plates and scattered
cells of every density, on grids at the edges of the block sizes, against the walk
cell by cell (a captured render, which takes no block occupancy)."""
import numpy as np
import pytest

from paper_2303_14827_gb300 import binding, scenes

pytestmark = pytest.mark.gpu


def grids(g):
    import torch
    a = (torch.arange(g, device="cuda", dtype=torch.float32) + 0.5) / g * 2 - 1
    z, y, x = a[:, None, None], a[None, :, None], a[None, None, :]
    r2 = x * x + y * y + z * z
    yield "ball", r2 < 0.81
    yield "ball off centre", (x - 0.4) ** 2 + (y + 0.3) ** 2 + z * z < 0.2
    yield "shell", (r2 < 0.81) & (r2 > 0.7)
    yield "half", x + 0.3 * y + 0.1 * z + 0 * r2 > 0.35
    yield "all but a tunnel", (x * x + y * y > 0.3) & (r2 < 9)
    yield "plates", ((torch.arange(g, device="cuda") % 9 == 4)[:, None, None]) & (r2 < 1.2)
    for d in (1e-4, 1e-3, 4e-3, 0.02, 0.3, 0.7):
        gen = torch.Generator("cuda").manual_seed(g)
        yield f"noise {d:g}", torch.rand((g, g, g), device="cuda", generator=gen) < d


@pytest.mark.parametrize("g", (31, 32, 63, 64, 95, 96, 97, 129, 200))
def test_blocks_equal_cells(g):
    import torch
    ctx = binding.dqj_create(0)
    stream = torch.cuda.Stream()
    try:
        for name, occ in grids(g):
            occ = occ.to(torch.uint8).reshape(-1).contiguous()
            for view in (dict(eye=[0.37, 0.23, 3.4], target=[0.05, -0.11, 0.02]), dict(eye=[0.3, 1.2, 0.9])):
                s = scenes.default_scene(width=203, height=117, **view)
                a, b = (binding.alloc_outputs(203, 117, stats=False) for _ in range(2))
                torch.cuda.synchronize()
                binding.dqj_render_voxels(ctx, s, g, occ, binding.outputs_of(a), stream.cuda_stream)
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    binding.dqj_render_voxels(ctx, s, g, occ, binding.outputs_of(b), stream.cuda_stream)
                graph.replay()
                torch.cuda.synchronize()
                for k in ("iter", "depth", "normal", "rgba"):
                    assert np.array_equal(a[k].cpu().numpy(), b[k].cpu().numpy()), (g, name, view, k)
    finally:
        binding.dqj_destroy(ctx)
