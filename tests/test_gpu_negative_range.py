"""Rays whose range reaches below 0 (minT < 0): the closest hit is the one with the lowest t."""
import numpy as np
import pytest

import oracle
import paper_2603_00292_gb300 as grt
from paper_2603_00292_gb300.objects import Geometry, device_tensor, hits_to_numpy, new_hits

pytestmark = pytest.mark.gpu


def _fans(n, nearer):
    """n triangles left and n right of the z axis; one of each touches the axis, with its lowest
    point, at -5 and `nearer` units in the last place below it."""
    low = np.float32(-5.0)
    lower = (np.array(low).view(np.uint32) + np.uint32(nearer)).view(np.float32)[()]
    v = []
    for side, z in ((-1.0, low), (1.0, lower)):
        v.append([[0, 0, z], [2 * side, 1, -4], [2 * side, -1, -4]])
        for k in range(n - 1):
            x, y = (2 + 0.1 * k) * side, 0.05 * k
            v.append([[x, y, -4.5], [x + 0.01, y, -4.5], [x, y + 0.01, -4.4]])
    return np.array(v, np.float32).reshape(-1, 3), np.arange(6 * n, dtype=np.uint32).reshape(-1, 3)


@pytest.mark.parametrize("nearer", [6, 7, 10, 1000])
@pytest.mark.parametrize("rays_n", [3, 1 << 20])
@pytest.mark.parametrize("fmt", [0, grt.GRT_BUILD_QUANTIZED_NODES, grt.GRT_BUILD_WIDE8_NODES])
def test_lowest_t_below_zero(gpu, fmt, rays_n, nearer):
    v, f = _fans(8, nearer)
    rays = np.zeros((rays_n, 8), np.float32)
    rays[:, 3], rays[:, 6], rays[:, 7] = -100.0, 1.0, 100.0
    S = oracle.Scene()
    S.add_instance(S.add_mesh(v, f))
    ref = S.trace(rays[:1], bvh=False)
    assert ref.prim[0] == 8
    g = Geometry(gpu, vertices=device_tensor(v), indices=device_tensor(f), build_flags=fmt).build()
    hits = new_hits(rays_n)
    grt.grtTraceClosest(gpu.handle, None, g.handle, device_tensor(rays), rays_n, hits)
    _, prim, t, _, _ = hits_to_numpy(hits)
    assert (prim == 8).all() and (t == np.float32(ref.t[0])).all()
    g.close()
