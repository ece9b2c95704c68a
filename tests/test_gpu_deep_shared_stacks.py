"""Closest hits with shared stacks whose size needs a kernel's opt-in (blocks of 256, depths
above 19), in any order of depths: a call with a smaller stack takes nothing from a later one."""
import pytest
import torch

import paper_2603_00292_gb300 as grt
import scenegen
from paper_2603_00292_gb300.objects import Geometry, device_tensor, new_hits, new_rays

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [50_000, 1 << 20])
@pytest.mark.parametrize("flags", [0, grt.GRT_BUILD_QUANTIZED_NODES])
@pytest.mark.parametrize("count", [False, True])
def test_a_smaller_stack_between_two_of_the_largest(gpu, flags, n, count):
    m = scenegen.terrain(40, 0.2)
    g = Geometry(gpu, vertices=device_tensor(m.vertices), indices=device_tensor(m.indices), build_flags=flags).build()
    rays = new_rays(n)
    grt.grtGenerateUniformRays(gpu.handle, [-1, -1, -1], [1, 1, 1], 5, n, rays)
    want = new_hits(n)
    grt.grtTraceClosest(gpu.handle, None, g.handle, rays, n, want)
    for depth in (32, 24, 32, 20, 19, 32):
        o = grt.trace_options(block_size=256, shared_depth=depth,
                              flags=grt.GRT_TRACE_FLAG_COUNT if count else 0)
        hits = new_hits(n)
        grt.grtTraceClosest(gpu.handle, None, g.handle, rays, n, hits, None, o)
        assert torch.equal(hits, want), depth
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
    g.close()
