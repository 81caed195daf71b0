"""dqj_render_voxels beside other work: during a stream capture elsewhere, on two
streams of one context at once, and on occupancies at any address."""
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


def test_two_streams_of_one_context():
    import torch
    ctx = binding.dqj_create(0)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    try:
        jobs = [(g, occupancy(g, d, g), view(eye=[0.37 + 0.1 * i, 0.23, 3.4]))
                for i, (g, d) in enumerate(((200, 0.0), (200, 1.0), (24, 0.1), (97, 1e-3), (129, 1e-4), (200, 1e-5)))]
        want = []
        for g, occ, s in jobs:
            t = binding.alloc_outputs(161, 121, stats=False)
            torch.cuda.synchronize()
            binding.dqj_render_voxels(ctx, s, g, occ, binding.outputs_of(t), streams[0].cuda_stream)
            torch.cuda.synchronize()
            want.append(planes(t))
        outs = [[binding.alloc_outputs(161, 121, stats=False) for _ in range(40)] for _ in jobs]
        torch.cuda.synchronize()
        for r in range(40):
            for i, (g, occ, s) in enumerate(jobs):
                binding.dqj_render_voxels(ctx, s, g, occ, binding.outputs_of(outs[i][r]),
                                          streams[(i + r // 2) % 2].cuda_stream)
        torch.cuda.synchronize()
        for i in range(len(jobs)):
            for r in range(40):
                assert same(planes(outs[i][r]), want[i]), (i, r)
    finally:
        binding.dqj_destroy(ctx)


@pytest.mark.parametrize("g", (24, 28, 96, 104))
@pytest.mark.parametrize("off", (1, 2, 4, 8))
def test_image_of_an_occupancy_at_any_address(g, off):
    import torch
    with binding.Renderer(0) as r:
        occ = occupancy(g, 1e-3, g)
        buf = torch.zeros(g ** 3 + 16, dtype=torch.uint8, device="cuda")
        moved = buf[off:off + g ** 3]
        moved.copy_(occ)
        got = []
        for o in (occ, moved):
            t = binding.alloc_outputs(161, 121, stats=False)
            binding.dqj_render_voxels(r.ctx, view(), g, o, binding.outputs_of(t), torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            got.append(planes(t))
        assert same(*got)


@pytest.mark.parametrize("g", (336, 337))
@pytest.mark.parametrize("off_occ,off_cnt", [(0, 2), (1, 0), (8, 16), (3, 6), (16, 16)])
def test_grid_at_any_address(g, off_occ, off_cnt):
    # offsets in bytes; nothing outside the grid is written
    import torch
    n = g ** 3
    s = scenes.default_scene(max_iter=14)
    with binding.Renderer(0) as r:
        st = torch.cuda.current_stream().cuda_stream
        occ = torch.empty(n, dtype=torch.uint8, device="cuda")
        cnt = torch.empty(n, dtype=torch.int16, device="cuda")
        binding.dqj_voxelize(r.ctx, s, g, occ, cnt, None, st)
        bo = torch.full((n + 64,), 77, dtype=torch.uint8, device="cuda")
        bc = torch.full((n + 32,), 77, dtype=torch.int16, device="cuda")
        mo, mc = bo[off_occ:off_occ + n], bc[off_cnt // 2:off_cnt // 2 + n]
        binding.dqj_voxelize(r.ctx, s, g, mo, mc, None, st)
        torch.cuda.synchronize()
        assert bool((mo == occ).all()) and bool((mc == cnt).all())
        assert bool((bo[:off_occ] == 77).all()) and bool((bo[off_occ + n:] == 77).all())
        assert bool((bc[:off_cnt // 2] == 77).all()) and bool((bc[off_cnt // 2 + n:] == 77).all())
