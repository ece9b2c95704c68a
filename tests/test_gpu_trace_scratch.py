"""The context's stack area: as much as the traces made so far need of it, and enough for a
captured trace of another kind over no more rays."""
import pytest
import torch

import paper_2603_00292_gb300 as grt
import scenegen
from paper_2603_00292_gb300.objects import Context, Geometry, device_tensor, new_hits, new_rays

pytestmark = pytest.mark.gpu
MIB = 1 << 20


def _terrain(ctx):
    m = scenegen.terrain(40, 0.2)
    return Geometry(ctx, vertices=device_tensor(m.vertices), indices=device_tensor(m.indices)).build()


def _rays(ctx, n):
    rays = new_rays(n)
    grt.grtGenerateUniformRays(ctx.handle, [-1, -1, -1], [1, 1, 1], 5, n, rays)
    return rays


def test_memory_of_a_first_trace(gpu):
    g = _terrain(gpu)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rays = _rays(gpu, 200_000)
    hits = new_hits(200_000)
    for n in (1, 200_000):  # loads the kernels
        grt.grtTraceClosest(gpu.handle, None, g.handle, rays, n, hits)
        grt.grtTraceAnyHit(gpu.handle, None, g.handle, rays, n, hits)
    torch.cuda.synchronize()
    for n, most in ((1, 2 * MIB), (100, 2 * MIB), (200_000, sms * 1024 * 64 * 4)):
        with Context(0) as ctx:
            torch.cuda.synchronize()
            before = torch.cuda.mem_get_info()[0]
            grt.grtTraceClosest(ctx.handle, None, g.handle, rays, n, hits)
            torch.cuda.synchronize()
            assert before - torch.cuda.mem_get_info()[0] <= most + 2 * MIB
    g.close()


@pytest.mark.parametrize("depth", [0, 100])
@pytest.mark.parametrize("warm, n", [(900_000, 1 << 20), (5000, 5000), (40, 40), (100_000, 1 << 20)])
def test_a_captured_trace_of_another_kind_finds_its_stacks(gpu, warm, n, depth):
    g = _terrain(gpu)
    rays = _rays(gpu, n)
    o = grt.trace_options(global_depth=depth)
    want, any_want = new_hits(n), new_hits(n)
    grt.grtTraceClosest(gpu.handle, None, g.handle, rays, n, want, None, o)
    grt.grtTraceAnyHit(gpu.handle, None, g.handle, rays, n, any_want, None, o)
    torch.cuda.synchronize()
    with Context(0) as ctx:
        hits, any_hits = new_hits(n), new_hits(n)
        grt.grtTraceClosest(ctx.handle, None, g.handle, rays, warm, hits, None, o)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            grt.grtTraceClosest(ctx.handle, None, g.handle, rays, n, hits, None, o)
            grt.grtTraceAnyHit(ctx.handle, None, g.handle, rays, n, any_hits, None, o)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(hits, want) and torch.equal(any_hits, any_want)
        assert grt.grtGetLastDeviceError(ctx.handle) == grt.GRT_SUCCESS
    g.close()
