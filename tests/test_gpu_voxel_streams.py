"""dqj_render_voxels beside other work: during a stream capture elsewhere."""
import numpy as np
import pytest

from paper_2303_14827_gb300 import binding, scenes

pytestmark = pytest.mark.gpu

PLANES = ("iter", "depth", "normal", "rgba")


def occupancy(g, density, seed):
    import torch
    gen = torch.Generator("cuda").manual_seed(seed)
    return (torch.rand(g ** 3, device="cuda", generator=gen) < density).to(torch.uint8)


def planes(t):
    return {k: t[k].cpu().numpy() for k in PLANES}


def same(a, b):
    return all(np.array_equal(a[k], b[k]) for k in PLANES)


def view(**kw):
    return scenes.default_scene(**dict(dict(width=161, height=121, eye=[0.37, 0.23, 3.4], target=[0.05, -0.11, 0.02]), **kw))


@pytest.mark.parametrize("first", (True, False))
def test_during_a_capture_on_another_stream(first):
    # first: the context's first such call falls into the capture
    import torch
    ctx = binding.dqj_create(0)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    try:
        occ = occupancy(100, 0.01, 3)
        s = view()
        a, b = (binding.alloc_outputs(161, 121, stats=False) for _ in range(2))
        x = torch.zeros(1000, device="cuda")
        torch.cuda.synchronize()
        if not first:
            binding.dqj_render_voxels(ctx, s, 100, occ, binding.outputs_of(a), s2.cuda_stream)
            torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s1):
            x.add_(1)
            binding.dqj_render_voxels(ctx, s, 100, occ, binding.outputs_of(a), s2.cuda_stream)
            x.add_(1)
        graph.replay()
        torch.cuda.synchronize()
        assert bool((x == 2).all())
        binding.dqj_render_voxels(ctx, s, 100, occ, binding.outputs_of(b), s2.cuda_stream)
        torch.cuda.synchronize()
        assert same(planes(a), planes(b))
    finally:
        binding.dqj_destroy(ctx)
