"""Builds around the sizes where one block, plain launches and a captured graph take over from
each other: the first builds of a description, those that replay its graph, and builds that
change it, equal the oracle bit for bit."""
import numpy as np
import pytest
import torch

import paper_2603_00292_gb300 as grt
from paper_2603_00292_gb300.objects import Geometry, device_tensor
from test_gpu_build import check_bit_exact

pytestmark = pytest.mark.gpu
SIZES = [1024, 1025, 1152, 1153, 1535, 1536, 1537, 2047, 2048, 2049]


def _boxes(n, seed):
    rng = np.random.default_rng([n, seed])
    c = rng.uniform(-1, 1, (n, 3))
    h = rng.uniform(0.0, 1e-2, (n, 3))
    return np.concatenate([c - h, c + h], axis=1).astype(np.float32)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("bits", [30, 63])
@pytest.mark.parametrize("flags", [0, grt.GRT_BUILD_WIDE8_NODES])
def test_builds_of_one_description(gpu, n, bits, flags):
    cases = [dict(boxes=_boxes(n, k)) for k in range(7)]  # the graph is captured for the fifth
    boxes = device_tensor(cases[0]["boxes"])
    g = Geometry(gpu, boxes=boxes, morton_bits=bits, build_flags=flags)
    for case in cases:  # other boxes in the same buffer
        boxes.copy_(device_tensor(case["boxes"]))
        g.build()
        check_bit_exact(g, case, bits)
    temps = [g.temp, torch.empty_like(g.temp)]
    for k in range(4):  # another description each time
        boxes.copy_(device_tensor(cases[k]["boxes"]))
        g.temp = temps[(k + 1) % 2]
        g.build()
        check_bit_exact(g, cases[k], bits)
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
    g.close()


@pytest.mark.parametrize("n", [1100, 2048])
def test_captured_by_the_caller_between_others(gpu, n):
    cases = [dict(boxes=_boxes(n, k)) for k in range(2)]
    boxes = device_tensor(cases[0]["boxes"])
    g = Geometry(gpu, boxes=boxes, morton_bits=30).build()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        g.build()
    for _ in range(6):
        boxes.copy_(device_tensor(cases[0]["boxes"]))
        g.build()
        check_bit_exact(g, cases[0], 30)
        boxes.copy_(device_tensor(cases[1]["boxes"]))
        graph.replay()
        check_bit_exact(g, cases[1], 30)
    g.close()
