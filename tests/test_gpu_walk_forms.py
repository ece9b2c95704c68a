"""Forms of the walk that depend on the number of rays (rays spread over the warps of a small
launch; phased or per-ray closest hits) give the same records, and slab tests hold for
directions with zero components and for rays that are not finite."""
import numpy as np
import pytest
import torch

import oracle
import paper_2603_00292_gb300 as grt
import scenegen
from parity import NONE, compare_any, compare_closest
from paper_2603_00292_gb300.objects import (FuncTable, Geometry, Scene, device_tensor, hits_to_numpy, new_hits,
                                            new_rays)

pytestmark = pytest.mark.gpu
FORMATS = {"plain": 0, "quantised": grt.GRT_BUILD_QUANTIZED_NODES, "wide8": grt.GRT_BUILD_WIDE8_NODES}


def _trace(ctx, rays, geom=None, scene=None, any_hit=False, table=None):
    hits = new_hits(rays.shape[0])
    f = grt.grtTraceAnyHit if any_hit else grt.grtTraceClosest
    f(ctx.handle, scene, geom, rays, rays.shape[0], hits, table)
    return hits


def _terrain(gpu, flags):
    m = scenegen.terrain(40, 0.2)
    return m, Geometry(gpu, vertices=device_tensor(m.vertices), indices=device_tensor(m.indices),
                       build_flags=flags).build()


@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("what", ["mesh", "spheres"])
def test_records_do_not_depend_on_the_number_of_rays(gpu, what, fmt):
    table = None
    if what == "mesh":
        _, g = _terrain(gpu, FORMATS[fmt])
    else:
        s = scenegen.spheres(3000, half=1.0, rmin=0.01, rmax=0.1, config=17)
        g = Geometry(gpu, boxes=device_tensor(scenegen.sphere_aabbs(s)), build_flags=FORMATS[fmt]).build()
        table = FuncTable(gpu)
        table.set(0, 0, grt.GRT_INTERSECT_SPHERE, device_tensor(s))
    n = (1 << 20) + 37  # the per-ray form; the pieces below take the phased one
    rays = new_rays(n)
    grt.grtGenerateUniformRays(gpu.handle, [-1, -1, -1], [1, 1, 1], 5, n, rays)
    for any_hit in (False, True):
        args = dict(geom=g.handle, any_hit=any_hit, table=table.handle if table else None)
        whole = _trace(gpu, rays, **args)
        pieces = torch.cat([_trace(gpu, rays[a:b].contiguous(), **args) for a, b in ((0, 600_000), (600_000, n))])
        assert torch.equal(whole, pieces)
        for k in (1, 2, 31, 33, 1000, 5003, 30_000):  # fewer than eight rays a warp
            assert torch.equal(_trace(gpu, rays[:k].contiguous(), **args), whole[:k])
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
    g.close()


def _axis_rays(n):
    """Rays with one or two zero direction components (of either sign), from random points."""
    rng = np.random.default_rng(23)
    d = rng.normal(size=(n, 3))
    d[np.arange(n), rng.integers(0, 3, n)] = 0.0
    half = rng.random(n) < 0.5
    d[half, rng.integers(0, 3, half.sum())] = -0.0
    d[(d == 0).all(1)] = [0.0, -1.0, -0.0]
    r = np.zeros((n, 8), np.float32)
    r[:, :3] = rng.uniform(-1.5, 1.5, (n, 3))
    r[:, 4:7] = d
    r[:, 7] = np.inf
    return r


@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("two_level", [False, True])
def test_zero_direction_components_match_oracle(gpu, fmt, two_level):
    m, g = _terrain(gpu, FORMATS[fmt])
    S = oracle.Scene()
    rays = _axis_rays(20_000)
    scene = None
    if two_level:
        q = np.array([[0, 0, 0, 1], [0, 0, np.sqrt(0.5), np.sqrt(0.5)]], np.float32)
        f = np.concatenate([q, np.ones((2, 3)), [[0, 0, 0], [0.3, 0.5, -0.2]]], axis=1).astype(np.float32)
        scene = Scene(gpu, [g.handle] * 2, device_tensor(f),
                      build_flags=FORMATS[fmt] if fmt == "wide8" else 0).build()
        mesh = S.add_mesh(m.vertices, m.indices)
        for k in range(2):
            S.add_instance(mesh, f[k])
    else:
        S.add_instance(S.add_mesh(m.vertices, m.indices))
    ref = S.trace(rays)
    args = dict(scene=scene.handle) if scene else dict(geom=g.handle)
    r = device_tensor(rays)
    compare_closest(hits_to_numpy(_trace(gpu, r, **args)), ref, S, rays, extent=3.0).check()
    compare_any(hits_to_numpy(_trace(gpu, r, any_hit=True, **args))[1], ref, S, rays, extent=3.0).check()
    if scene:
        scene.close()
    g.close()


@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("two_level", [False, True])
def test_rays_that_are_not_finite_miss(gpu, fmt, two_level):
    m, g = _terrain(gpu, FORMATS[fmt])
    scene = None
    if two_level:
        f = np.array([[0, 0, 0, 1, 1, 1, 1, 0, 0, 0]], np.float32)
        scene = Scene(gpu, [g.handle], device_tensor(f), build_flags=FORMATS[fmt] if fmt == "wide8" else 0).build()
    bad = [np.nan, np.inf, -np.inf]
    rows = [[0.1, 1.0, 0.2, 0, 0, -1, 0, np.inf]]  # an ordinary hit among them
    for x in bad:
        rows += [[0, 1, 0, 0, x, x, x, np.inf], [0, 1, 0, 0, x, -1, 0, np.inf], [x, 1, 0, 0, 0, -1, 0, np.inf],
                 [x, x, x, 0, 0, -1, 0, np.inf]]
    rays = device_tensor(np.array(rows, np.float32))
    args = dict(scene=scene.handle) if scene else dict(geom=g.handle)
    for any_hit in (False, True):
        prim = hits_to_numpy(_trace(gpu, rays, any_hit=any_hit, **args))[1]
        assert prim[0] != NONE and (prim[1:] == NONE).all()
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
    if scene:
        scene.close()
    g.close()


@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("two_level", [False, True])
def test_rays_in_the_planes_of_boxes_hit_inclusive_edges(gpu, fmt, two_level):
    """Rays straight down on the vertices and edges of a flat grid whose far sides lie at 0: they
    lie in the planes of the boxes, and edges belong to their triangles."""
    m = scenegen.terrain(8, 0.0)
    v = m.vertices.copy()
    v[:, [0, 2]] -= 1.0  # [-2, 0]^2, multiples of 1/4
    g = Geometry(gpu, vertices=device_tensor(v), indices=device_tensor(m.indices), build_flags=FORMATS[fmt]).build()
    k = np.concatenate([np.arange(9) / 4.0 - 2.0, [-0.0]]).astype(np.float32)
    x, z = (a.ravel() for a in np.meshgrid(k, np.concatenate([k, k[:8] + 0.125])))
    rays = np.zeros((2 * x.size, 8), np.float32)
    rays[:, 0], rays[:, 2] = np.tile(x, 2), np.tile(z, 2)
    rays[:, 1] = 1.0
    rays[:, 5] = -1.0
    rays[x.size:, [4, 6]] = -0.0
    rays[:, 7] = np.inf
    scene = None
    if two_level:
        f = np.array([[0, 0, 0, 1, 1, 1, 1, 0, 0, 0]], np.float32)
        scene = Scene(gpu, [g.handle], device_tensor(f), build_flags=FORMATS[fmt] if fmt == "wide8" else 0).build()
    args = dict(scene=scene.handle) if scene else dict(geom=g.handle)
    r = device_tensor(rays)
    for any_hit in (False, True):
        _, prim, t, _, _ = hits_to_numpy(_trace(gpu, r, any_hit=any_hit, **args))
        assert (prim != NONE).all() and np.all(np.abs(t - 1.0) <= 1e-5)
    big = r.repeat(-(-(1 << 20) // r.shape[0]), 1)[:1 << 20].contiguous()  # the per-ray form
    assert (hits_to_numpy(_trace(gpu, big, **args))[1] != NONE).all()
    if scene:
        scene.close()
    g.close()


@pytest.mark.parametrize("any_hit", [False, True])
@pytest.mark.parametrize("n", [5000, 50_000, 1 << 20])
def test_a_callers_stack_buffer_bounds_the_grid(gpu, n, any_hit):
    _, g = _terrain(gpu, 0)
    rays = new_rays(n)
    grt.grtGenerateUniformRays(gpu.handle, [-1, -1, -1], [1, 1, 1], 9, n, rays)
    whole = _trace(gpu, rays, geom=g.handle, any_hit=any_hit)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = min(-(-n // 128), sms * (5 if any_hit else 4))
    f = grt.grtTraceAnyHit if any_hit else grt.grtTraceClosest
    for size, accepted in ((blocks * 128 * 64 * 4, True), (blocks * 128 * 64 * 4 - 256, False)):
        stack = torch.empty(size, dtype=torch.uint8, device="cuda")
        o = grt.trace_options(global_stack=stack, global_stack_bytes=size)
        hits = new_hits(n)
        if accepted:
            f(gpu.handle, None, g.handle, rays, n, hits, None, o)
            assert torch.equal(hits, whole)
        else:
            with pytest.raises(grt.GrtError):
                f(gpu.handle, None, g.handle, rays, n, hits, None, o)
    g.close()
