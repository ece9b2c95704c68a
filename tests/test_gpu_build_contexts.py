"""Builds of one geometry through several contexts: a build belongs to the context it is called
with, also where another one built the same buffers before and is gone."""
import numpy as np
import pytest
import torch

import paper_2603_00292_gb300 as grt
from paper_2603_00292_gb300.objects import Context, Geometry, device_tensor
from test_gpu_build import check_bit_exact

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, grt.GRT_BUILD_WIDE8_NODES])
def test_rebuilds_through_other_contexts(gpu, flags):
    n = 20_001
    rng = np.random.default_rng(n)
    c = rng.uniform(-1, 1, (n, 3))
    case = dict(boxes=np.concatenate([c - 1e-3, c + 1e-3], axis=1).astype(np.float32))
    g = Geometry(gpu, boxes=device_tensor(case["boxes"]), build_flags=flags)
    for _ in range(3):
        with Context(0) as other:
            for ctx in (gpu, other, other, gpu):
                g.ctx = ctx
                g.build()
                assert grt.grtGetLastDeviceError(ctx.handle) == grt.GRT_SUCCESS
        g.ctx = gpu  # the other context is gone
        g.build()
        torch.cuda.synchronize()
        check_bit_exact(g, case, 30)
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
    g.close()
