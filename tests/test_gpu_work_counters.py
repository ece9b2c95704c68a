"""Work counters of the traces: no call depends on what an earlier launch left in its slot, and
captured launches keep theirs beside launches issued at once."""
import numpy as np
import pytest
import torch

import paper_2603_00292_gb300 as grt
import scenegen
from paper_2603_00292_gb300.objects import Context, Geometry, Scene, device_tensor, device_view, new_hits, new_rays

pytestmark = pytest.mark.gpu
# the context's device workspace: error word and statistics (256 bytes), then 256 counters of
# launches issued at once and 1,024 of captured ones, 8 bytes each
COUNTERS = (256, 1280 * 8)


def _leave_traces(ctx, geom):
    """Fills every counter as launches would that shared their slots and left them so."""
    at = grt.grtGetDeviceTarget(ctx.handle, geom=geom).deviceError + COUNTERS[0]
    device_view(at, COUNTERS[1]).fill_(0x3F)


@pytest.fixture
def own():
    with Context(0) as ctx:
        m = scenegen.terrain(48, 0.2)
        v, f = device_tensor(m.vertices), device_tensor(m.indices)
        g = Geometry(ctx, vertices=v, indices=f).build()
        fr = scenegen.random_frames(4, seed=3)
        sc = Scene(ctx, [g.handle] * 4, device_tensor(fr.packed())).build()
        yield ctx, g, sc, v, f
        torch.cuda.synchronize()
        sc.close()
        g.close()


def _calls(ctx, g, sc, v, f, n):
    """One call of every kind that takes work from a counter; its results."""
    rays = new_rays(n)
    grt.grtGenerateUniformRays(ctx.handle, [-1, -1, -1], [1, 1, 1], 11, n, rays)
    out = []
    for fn in (grt.grtTraceClosest, grt.grtTraceAnyHit, grt.grtTraceClosestNoAlloc):
        for scene, geom in ((None, g.handle), (sc.handle, None)):
            h = torch.full_like(new_hits(n), -1)
            fn(ctx.handle, scene, geom, rays, n, h)
            out.append(h)
    ao = torch.zeros(n, device="cuda")
    grt.grtTraceAmbientOcclusion(ctx.handle, sc.handle, rays, out[1], n, 4, 7, 0.5, ao)
    out.append(ao)
    colours = torch.rand((v.shape[0], 3), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    light = torch.tensor([0.3, 1.0, 0.2], device="cuda")
    image, vis = torch.zeros((n, 3), device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda")
    grt.grtShadeLambert(ctx.handle, g.handle, rays, out[0], n, f, v, colours, light, image, vis)
    out += [image, vis]
    gc, gl, gp = torch.zeros_like(colours), torch.zeros(3, device="cuda"), torch.zeros_like(v)
    ones = torch.full((n, 3), 1.0 / n, device="cuda")
    grt.grtShadeLambertBackward(ctx.handle, g.handle, rays, out[0], vis, n, f, v, colours, light, ones, gc, gl, gp)
    return out, [gc, gl, gp]


@pytest.mark.parametrize("n", [900, 200_000, (1 << 20) + 5])
def test_calls_do_not_depend_on_the_counters_they_find(own, n):
    ctx, g = own[:2]
    want, grads = _calls(*own, n)
    assert (want[0][:, 1] != -1).sum() > n // 20
    assert torch.equal(want[0], want[4]) and torch.equal(want[1], want[5])  # with and without allocation
    for _ in range(2):
        torch.cuda.synchronize()
        _leave_traces(ctx, g.handle)
        got, back = _calls(*own, n)
        for a, b in zip(got, want):
            assert torch.equal(a, b)
        for a, b in zip(back, grads):  # atomic sums in any order
            assert (a - b).abs().max() <= 1e-4 * max(float(b.abs().max()), 1e-6)
    assert grt.grtGetLastDeviceError(ctx.handle) == grt.GRT_SUCCESS


def test_captured_traces_between_many_issued_at_once(own):
    ctx, g = own[:2]
    n = 60_000
    rays = new_rays(n)
    grt.grtGenerateUniformRays(ctx.handle, [-1, -1, -1], [1, 1, 1], 12, n, rays)
    size = grt.grtGetTraceGlobalStackSize(ctx.handle)
    stacks = [torch.empty(size, dtype=torch.uint8, device="cuda") for _ in range(2)]
    opts = [grt.trace_options(global_stack=s, global_stack_bytes=size) for s in stacks]
    want, eager, replayed = new_hits(n), new_hits(n), new_hits(n)
    grt.grtTraceClosest(ctx.handle, None, g.handle, rays, n, want)
    eager.copy_(want), replayed.copy_(want)
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph):
        grt.grtTraceClosest(ctx.handle, None, g.handle, rays, n, replayed, None, opts[0])
    for i in range(600):
        grt.grtTraceClosest(ctx.handle, None, g.handle, rays, n, eager, None, opts[1], side)
        if i % 20 == 7:  # beside the eager ones, which wait for nothing
            graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(eager, want) and torch.equal(replayed, want)
    assert grt.grtGetLastDeviceError(ctx.handle) == grt.GRT_SUCCESS
