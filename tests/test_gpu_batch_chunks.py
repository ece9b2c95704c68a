"""Work items of a batch sized by the batch (traceChunk, buildChunk left open) give the hit
records of any fixed sizes: ray counts around an item's, scenes built by one block and not."""
import numpy as np
import pytest
import torch

import paper_2603_00292_gb300 as grt
import scenegen
from paper_2603_00292_gb300.objects import Batch, Geometry, device_tensor, new_hits, new_rays

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1, 40])
def test_items_sized_by_the_batch_change_no_record(gpu, scale):
    rays_of = [1, 511, 512, 513, 1025, 4096]
    prims_of = [3, 1000, 8192, 8193, 9216, 9217]

    def batch(**options):
        scenes = []
        for k, (n, r) in enumerate(zip(prims_of, rays_of)):
            s = scenegen.soup_scene(k, seed=77, nmin=n, nmax=n, rmin=16, rmax=16)
            g = Geometry(gpu, vertices=device_tensor(s.mesh.vertices), indices=device_tensor(s.mesh.indices))
            rays = new_rays(r * scale)
            grt.grtGenerateUniformRays(gpu.handle, s.lo, s.hi, k, r * scale, rays)
            scenes.append((g, rays, new_hits(r * scale)))
        b = Batch(gpu, scenes, grt.batch_options(**options)).run()
        torch.cuda.synchronize()
        hits = [h.cpu().numpy() for _, _, h in scenes]
        items = b.info().itemCount
        b.close()
        for g, _, _ in scenes:
            g.close()
        return hits, items

    sized, many = batch()
    fixed, few = batch(trace_chunk=16384, build_chunk=16384)
    assert many > few
    assert all(np.array_equal(a, b) for a, b in zip(sized, fixed))
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
