"""Rays with zero direction components far from the origin of coordinates, where the product
of the origin and a reciprocal direction leaves the range of a float32 (from 2^22 on at a
reciprocal of 2^106), compared with the oracle; rays in the planes of boxes whatever the
length of their direction; and the work of rays with short directions."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_2603_00292_gb300 as grt
import scenegen
from paper_2603_00292_gb300.objects import (Batch, Geometry, Scene, device_tensor, hits_to_numpy, new_hits)
from parity import NONE, compare_any, compare_closest
from test_gpu_device_api import user_lib  # noqa: F401 (a fixture)

pytestmark = pytest.mark.gpu
FORMATS = {"plain": 0, "quantised": grt.GRT_BUILD_QUANTIZED_NODES, "wide8": grt.GRT_BUILD_WIDE8_NODES}
SHIFTS = [4194304.0, -4194304.0, 5e6, -5e6, 1e8, -1e8]


def _far_case(shift, n=20_000):
    """A terrain a quarter of `shift` in half size, moved by it along every axis, and rays with
    one or two zero components (of either sign) from points around it."""
    half = abs(shift) / 4
    m = scenegen.terrain(40, 0.2)
    at = np.array([shift, -shift, shift])
    v = (m.vertices.astype(np.float64) * half + at).astype(np.float32)
    rng = np.random.default_rng(31)
    d = rng.normal(size=(n, 3))
    d[np.arange(n), rng.integers(0, 3, n)] = 0.0
    two = rng.random(n) < 0.5
    d[two, rng.integers(0, 3, two.sum())] = -0.0
    d[(d == 0).all(1)] = [0.0, -1.0, -0.0]
    rays = np.zeros((n, 8), np.float32)
    rays[:, :3] = rng.uniform(-1.5, 1.5, (n, 3)) * [half, 0.3 * half, half] + at
    rays[:, 4:7] = d
    rays[:, 7] = np.where(rng.random(n) < 0.7, np.inf, 4 * half)
    return v, m.indices, rays, 3 * half


def _trace(gpu, rays, any_hit=False, geom=None, scene=None):
    hits = new_hits(rays.shape[0])
    (grt.grtTraceAnyHit if any_hit else grt.grtTraceClosest)(gpu.handle, scene, geom, rays, rays.shape[0], hits)
    return hits_to_numpy(hits)


@pytest.mark.parametrize("shift", SHIFTS)
@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("two_level", [False, True])
def test_far_axis_aligned_rays_match_oracle(gpu, two_level, fmt, shift):
    v, f, rays, extent = _far_case(shift)
    g = Geometry(gpu, vertices=device_tensor(v), indices=device_tensor(f), build_flags=FORMATS[fmt]).build()
    S = oracle.Scene()
    mesh = S.add_mesh(v, f)
    scene = None
    if two_level:
        frames = np.array([[0, 0, 0, 1, 1, 1, 1, 0, 0, 0], [0, 0, 0, 1, 1, 1, 1, extent / 4, 0, -extent / 8]], np.float32)
        scene = Scene(gpu, [g.handle] * 2, device_tensor(frames), build_flags=FORMATS[fmt] if fmt == "wide8" else 0).build()
        for k in range(2):
            S.add_instance(mesh, frames[k])
    else:
        S.add_instance(mesh)
    S.build()
    ref = S.trace(rays)
    assert (ref.prim != NONE).mean() > 0.1
    args = dict(scene=scene.handle) if scene else dict(geom=g.handle)
    r = device_tensor(rays)
    compare_closest(_trace(gpu, r, **args), ref, S, rays, extent=extent).check()
    compare_any(_trace(gpu, r, any_hit=True, **args)[1], ref, S, rays, extent=extent).check()
    if not two_level:  # the form of large launches
        big = r.repeat(-(-(1 << 20) // r.shape[0]), 1).contiguous()
        many = _trace(gpu, big, **args)
        compare_closest([a[:len(rays)] for a in many], ref, S, rays, extent=extent).check()
    k, n = 4, 2000  # every hit, through the library
    hits, counts = new_hits(n * k), torch.zeros(n, dtype=torch.int32, device="cuda")
    grt.grtTraceAllHits(gpu.handle, scene.handle if scene else None, None if scene else g.handle, r[:n], n, hits, k, counts)
    compare_any(np.where(counts.cpu().numpy() > 0, 0, NONE), _head(ref, n), S, rays[:n], extent=extent).check()
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
    if scene:
        scene.close()
    g.close()


class _Head:
    pass


def _head(ref, n):
    h = _Head()
    h.prim, h.t = ref.prim[:n], ref.t[:n]
    return h


@pytest.mark.parametrize("shift", [4194304.0, -1e8])
def test_far_axis_aligned_rays_in_a_batch_and_a_user_kernel(gpu, user_lib, shift):  # noqa: F811
    v, f, rays, extent = _far_case(shift)
    S = oracle.Scene()
    S.add_instance(S.add_mesh(v, f))
    S.build()
    ref = S.trace(rays)
    r = device_tensor(rays)
    g = Geometry(gpu, vertices=device_tensor(v), indices=device_tensor(f))
    hits = new_hits(len(rays))
    b = Batch(gpu, [(g, r, hits)], grt.batch_options()).run()
    torch.cuda.synchronize()
    compare_closest(hits_to_numpy(hits), ref, S, rays, extent=extent).check()
    T = grt.grtGetDeviceTarget(gpu.handle, geom=g.handle)
    for any_hit in (0, 1):
        hits.fill_(0)
        assert user_lib.userTraceLaunch(ctypes.byref(T), r.data_ptr(), len(rays), hits.data_ptr(), any_hit,
                                        torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        got = hits_to_numpy(hits)
        if any_hit:
            compare_any(got[1], ref, S, rays, extent=extent).check()
        else:
            compare_closest(got, ref, S, rays, extent=extent).check()
    b.close()
    g.close()


@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("two_level", [False, True])
@pytest.mark.parametrize("length, height", [(1.0, 1e9), (1e-4, 1.0), (1e-8, 1e4), (1e-12, 1.0), (1e-12, 1e8), (1e-20, 1e3),
                                            (1e-30, 1.0)])
def test_rays_in_box_planes_hit_with_directions_of_any_length(gpu, two_level, fmt, length, height):
    """Straight down on the vertices and edges of a flat grid in [-2, 0]^2: boxes have planes at 0,
    in which rays lie; edges belong to their triangles."""
    m = scenegen.terrain(8, 0.0)
    v = m.vertices.copy()
    v[:, [0, 2]] -= 1.0
    g = Geometry(gpu, vertices=device_tensor(v), indices=device_tensor(m.indices), build_flags=FORMATS[fmt]).build()
    k = np.concatenate([np.arange(9) / 4.0 - 2.0, [-0.0]]).astype(np.float32)
    x, z = (a.ravel() for a in np.meshgrid(k, np.concatenate([k, k[:8] + 0.125])))
    rays = np.zeros((2 * x.size, 8), np.float32)
    rays[:, 0], rays[:, 2] = np.tile(x, 2), np.tile(z, 2)
    rays[:, 1] = height
    rays[:, 5] = -length
    rays[x.size:, [4, 6]] = -0.0
    rays[:, 7] = np.inf
    scene = None
    if two_level:
        f = np.array([[0, 0, 0, 1, 1, 1, 1, 0, 0, 0]], np.float32)
        scene = Scene(gpu, [g.handle], device_tensor(f), build_flags=FORMATS[fmt] if fmt == "wide8" else 0).build()
    args = dict(scene=scene.handle) if scene else dict(geom=g.handle)
    r = device_tensor(rays)
    t = np.float64(np.float32(height)) / np.float64(np.float32(length))
    for any_hit in (False, True):
        got = _trace(gpu, r, any_hit=any_hit, **args)
        assert (got[1] != NONE).all() and np.all(np.abs(got[2] - t) <= 1e-5 * t)
    if scene:
        scene.close()
    g.close()


@pytest.mark.parametrize("fmt", list(FORMATS))
@pytest.mark.parametrize("two_level", [False, True])
@pytest.mark.parametrize("any_hit", [False, True])
def test_short_and_zero_directions_are_culled(gpu, fmt, two_level, any_hit):
    """Rays along an axis visit the same nodes whatever the length of their direction (to 2^-39 of
    the mesh in width), rays without one in a geometry those around their origins."""
    m = scenegen.terrain(64, 0.2)
    g = Geometry(gpu, vertices=device_tensor(m.vertices), indices=device_tensor(m.indices), build_flags=FORMATS[fmt]).build()
    scene = None
    if two_level:
        f = np.array([[0, 0, 0, 1, 1, 1, 1, 0, 0, 0]], np.float32)
        scene = Scene(gpu, [g.handle], device_tensor(f), build_flags=FORMATS[fmt] if fmt == "wide8" else 0).build()
    args = (scene.handle, None) if scene else (None, g.handle)
    n = 4000
    rng = np.random.default_rng(3)
    rays = np.zeros((n, 8), np.float32)
    rays[:, :3] = rng.uniform(-0.99, 0.99, (n, 3)) * [1, 0, 1] + [0, 1, 0]
    rays[:, 7] = np.inf
    hits = new_hits(n)

    def nodes(length):
        rays[:, 5] = -length
        grt.grtGetTraceStatistics(gpu.handle)  # reads and clears
        f = grt.grtTraceAnyHit if any_hit else grt.grtTraceClosest
        f(gpu.handle, *args, device_tensor(rays), n, hits, None, grt.trace_options(flags=grt.GRT_TRACE_FLAG_COUNT))
        found = (hits_to_numpy(hits)[1] != NONE).sum()
        return grt.grtGetTraceStatistics(gpu.handle)["nodesVisited"] / n, found

    want, all_hit = nodes(1.0)
    assert all_hit == n
    for length in (1e-6, 1e-9, 1e-12):
        visited, found = nodes(length)
        assert found == n and visited <= 1.1 * want, (length, visited, want)
    if not two_level:  # an instance's boxes are widened without end for a ray that never leaves them
        rays[:, 1] = 0.0  # among the triangles
        visited, found = nodes(0.0)
        assert found == 0 and visited <= 4 * want, (visited, want)
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
    if scene:
        scene.close()
    g.close()
