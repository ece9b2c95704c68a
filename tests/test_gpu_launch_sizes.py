"""Traces and shading at the sizes where the launch changes (fewer lanes than a warp, full warps in
as many blocks as they fill, more warps with fewer registers each) give the records of the same
rays in another launch."""
import pytest
import torch

import paper_2603_00292_gb300 as grt
import scenegen
from paper_2603_00292_gb300.objects import Geometry, Scene, device_tensor, new_hits, new_rays

pytestmark = pytest.mark.gpu
FORMATS = {"plain": 0, "quantised": grt.GRT_BUILD_QUANTIZED_NODES, "wide8": grt.GRT_BUILD_WIDE8_NODES}


def _edges():
    """Rays at which a grid of 16, 20, 24, 28 or 32 warps an SM has eight for each, and the launch
    sizes of the forms with more warps."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    at = [8 * sms * w for w in (16, 20, 24, 28, 32)] + [1 << 18]
    return sorted({n + d for n in at for d in (-1, 0, 1)} | {127, 129, 5000})


@pytest.mark.parametrize("fmt", list(FORMATS))
def test_records_at_the_edges_of_launch_sizes(gpu, fmt):
    m = scenegen.terrain(40, 0.2)
    v, f = device_tensor(m.vertices), device_tensor(m.indices)
    g = Geometry(gpu, vertices=v, indices=f, build_flags=FORMATS[fmt]).build()
    fr = scenegen.random_frames(4, seed=3)
    sc = Scene(gpu, [g.handle] * 4, device_tensor(fr.packed()), build_flags=FORMATS[fmt] if fmt == "wide8" else 0).build()
    n = (1 << 18) + 4000
    rays = new_rays(n)
    grt.grtGenerateUniformRays(gpu.handle, [-1, -1, -1], [1, 1, 1], 5, n, rays)
    colours = torch.rand((v.shape[0], 3), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    light = torch.tensor([0.3, 1.0, 0.2], device="cuda")

    def run(k):
        out = []
        for fn in (grt.grtTraceClosest, grt.grtTraceAnyHit):
            for args in ((None, g.handle), (sc.handle, None)):
                h = new_hits(k)
                fn(gpu.handle, *args, rays, k, h)
                out.append(h)
        image, vis = torch.zeros((k, 3), device="cuda"), torch.zeros(k, dtype=torch.uint8, device="cuda")
        grt.grtShadeLambert(gpu.handle, g.handle, rays, out[0], k, f, v, colours, light, image, vis)
        return out + [image, vis]

    whole = run(n)
    assert (whole[0][:, 1] != -1).sum() > n // 20 and whole[5].sum() > n // 50
    for k in _edges():
        for a, b in zip(run(k), whole):
            assert torch.equal(a, b[:k]), k
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
    sc.close()
    g.close()
