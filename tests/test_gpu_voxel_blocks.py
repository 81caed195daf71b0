"""The grid image by blocks (voxel_render_blocks_kernel) against the walk cell by
cell (a captured render, which takes no block occupancy): every plane equal, on
grids whose sides straddle block sizes, with empty, sparse, dense and full
occupancy, cameras on and off the grid's symmetry axes, grazing an edge and
inside the box."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g", (24, 25, 31, 95, 96, 97, 100, 129))
def test_blocks_equal_cells(g):
    import torch

    from paper_2303_14827_gb300 import binding, scenes

    ctx = binding.dqj_create(0)
    stream = torch.cuda.Stream()
    try:
        for seed, density in enumerate((0.0, 2e-4, 0.05, 1.0)):
            gen = torch.Generator("cuda").manual_seed(seed + g)
            occ = (torch.rand(g ** 3, device="cuda", generator=gen) < density).to(torch.uint8)
            for view in (dict(), dict(eye=[0.37, 0.23, 3.4], target=[0.05, -0.11, 0.02]),
                         dict(eye=[2.0, 2.0, 3.0], target=[-2.0, -2.0, -2.0]), dict(eye=[0.3, 1.2, 0.9]),
                         dict(eye=[30.0, 21.0, 25.0], fov_y_deg=9.0), dict(eye=[9.0, 9.0, 9.0])):
                s = scenes.default_scene(width=161, height=121, **view)
                a, b = (binding.alloc_outputs(161, 121, stats=False) for _ in range(2))
                torch.cuda.synchronize()
                with torch.cuda.stream(stream):
                    binding.dqj_render_voxels(ctx, s, g, occ, binding.outputs_of(a), stream.cuda_stream)
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    binding.dqj_render_voxels(ctx, s, g, occ, binding.outputs_of(b), stream.cuda_stream)
                graph.replay()
                torch.cuda.synchronize()
                for k in ("iter", "depth", "normal", "rgba"):
                    assert np.array_equal(a[k].cpu().numpy(), b[k].cpu().numpy()), (g, density, view, k)
    finally:
        binding.dqj_destroy(ctx)
