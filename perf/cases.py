"""The work that a user of this framework has it do, as cases that can be timed and compared.

Five kinds of call, each through the public entry points of paper_2603_00292_gb300:

  build    one bottom-level BVH build (a mesh or an AABB list that changes every frame)
  trace    closest hit (and any hit) of a ray buffer against one geometry or a two-level scene
  ao       fused ambient occlusion over primary hits of a two-level scene
  lambert  differentiable shading: forward, loss and backward
  batch    many uneven triangle soups built and traced in one captured launch

Inputs are synthetic and made on the GPU from the seed alone.
"""
import math

import torch

import paper_2603_00292_gb300 as grt
from paper_2603_00292_gb300 import objects, shading

_context = None


def _ctx():
    """One library context per process, as a program keeps it."""
    global _context
    if _context is None:
        _context = objects.Context(0)
    return _context


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest mesh of the repository's workloads rebuilt: all latency and launches
        {"name": "build_icosphere", "kind": "build", "shape": "icosphere", "size": 3, "wide8": False},
        # the benchmark's terrain, 131,072 triangles, with the 8-wide nodes its traces read
        {"name": "build_terrain", "kind": "build", "shape": "terrain", "size": 256, "wide8": True},
        # a large unstructured mesh with 63-bit codes, an odd number of triangles
        {"name": "build_soup", "kind": "build", "shape": "soup", "size": 1234567, "wide8": False},
        # a million custom primitives given by their boxes
        {"name": "build_spheres", "kind": "build", "shape": "spheres", "size": 1000000, "wide8": False},
        # a picking-sized query on a small mesh: launches and the longest ray
        {"name": "trace_small", "kind": "trace", "shape": "icosphere", "size": 3, "instances": 0, "width": 96,
         "height": 54, "distance": 3.0, "wide8": False},
        # one image of one small mesh
        {"name": "trace_icosphere", "kind": "trace", "shape": "icosphere", "size": 3, "instances": 0, "width": 512,
         "height": 512, "distance": 3.0, "wide8": False},
        # primary rays of the benchmark's instanced scene seen from afar: most rays miss
        {"name": "trace_terrain_far", "kind": "trace", "shape": "terrain", "size": 256, "instances": 64,
         "width": 1920, "height": 1080, "distance": 1.5, "wide8": True},
        # the same scene filling an odd-sized image, through the default 4-wide nodes
        {"name": "trace_terrain_near", "kind": "trace", "shape": "terrain", "size": 256, "instances": 64,
         "width": 1279, "height": 719, "distance": 0.35, "wide8": False},
        # the benchmark's ambient occlusion: incoherent short any-hit rays
        {"name": "ao_terrain", "kind": "ao", "shape": "terrain", "size": 256, "instances": 64, "width": 1920,
         "height": 1080, "distance": 1.5, "samples": 8, "wide8": True},
        # a million custom spheres under random rays, closest hit and any hit of each
        {"name": "trace_spheres", "kind": "trace", "shape": "spheres", "size": 1000000, "instances": 0,
         "rays": 4194304, "wide8": False},
        # one optimisation step through differentiable shading at 1080p
        {"name": "lambert_step", "kind": "lambert", "size": 3, "width": 1920, "height": 1080, "store": True},
        # many uneven scenes, each built and traced, in one launch
        {"name": "batch_soups", "kind": "batch", "scenes": 24, "most": 300000, "most_rays": 262144},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "trace", "trace", "trace", "ao", "lambert", "batch"])
    wide8 = rng.random() < 0.5
    if kind == "build":
        shape = rng.choice(["terrain", "soup", "spheres"])
        size = _log(rng, 16, 256) if shape == "terrain" else _log(rng, 1000, 1000000)
        return {"kind": kind, "shape": shape, "size": size, "wide8": wide8}
    image = {"width": _log(rng, 96, 1900), "height": _log(rng, 54, 1000)}
    scene = {"shape": "terrain", "size": _log(rng, 32, 256), "instances": rng.randint(2, 64)}
    if kind == "ao":
        return {"kind": kind, **scene, **image, "distance": 1.5, "samples": rng.randint(1, 8), "wide8": wide8}
    if kind == "lambert":
        return {"kind": kind, "size": rng.randint(2, 4), **image, "store": rng.random() < 0.7}
    if kind == "batch":
        return {"kind": kind, "scenes": rng.randint(6, 24), "most": _log(rng, 10000, 250000),
                "most_rays": _log(rng, 16384, 200000)}
    what = rng.choice(["icosphere", "terrain", "spheres"])
    if what == "spheres":
        return {"kind": kind, "shape": what, "size": _log(rng, 1000, 1000000), "instances": 0,
                "rays": _log(rng, 4096, 3000000), "wide8": wide8}
    if what == "icosphere":
        return {"kind": kind, "shape": what, "size": rng.randint(2, 5), "instances": 0, **image,
                "distance": rng.uniform(2.0, 5.0), "wide8": wide8}
    return {"kind": kind, **scene, **image, "distance": rng.uniform(0.35, 1.5), "wide8": wide8}


# ---------------------------------------------------------------- inputs, from the seed alone
def _rng(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFFFFFFFFFF)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _unit(g, n):
    z = 1.0 - 2.0 * _rand(g, n)
    phi = 2.0 * math.pi * _rand(g, n)
    s = (1.0 - z * z).clamp_min(0.0).sqrt()
    return torch.stack([s * phi.cos(), s * phi.sin(), z], 1)


def _turn(g):
    """A uniformly random rotation matrix."""
    return _matrix(_quaternions(g, 1))[0]


def _quaternions(g, n):
    u = _rand(g, n, 3)
    a, b, p, q = (1.0 - u[:, 0]).sqrt(), u[:, 0].sqrt(), 2.0 * math.pi * u[:, 1], 2.0 * math.pi * u[:, 2]
    return torch.stack([a * p.sin(), a * p.cos(), b * q.sin(), b * q.cos()], 1)


def _matrix(q):
    x, y, z, w = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    rows = [1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
            2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
            2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]
    return torch.stack(rows, 1).reshape(-1, 3, 3)


def _icosphere(level, g):
    """Unit icosphere, randomly turned: float32 vertices, int32 triangles."""
    p = (1.0 + math.sqrt(5.0)) / 2.0
    v = torch.tensor([(-1, p, 0), (1, p, 0), (-1, -p, 0), (1, -p, 0), (0, -1, p), (0, 1, p), (0, -1, -p), (0, 1, -p),
                      (p, 0, -1), (p, 0, 1), (-p, 0, -1), (-p, 0, 1)], dtype=torch.float64, device="cuda")
    v = v / v.norm(dim=1, keepdim=True)
    f = torch.tensor([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2),
                      (10, 7, 6), (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5),
                      (2, 4, 11), (6, 2, 10), (8, 6, 7), (9, 8, 1)], device="cuda")
    for _ in range(level):
        edges = torch.cat([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]).sort(1).values
        edges, where = torch.unique(edges, dim=0, return_inverse=True)
        mid = v[edges[:, 0]] + v[edges[:, 1]]
        ab, bc, ca = (where + v.shape[0]).reshape(3, -1)
        v = torch.cat([v, mid / mid.norm(dim=1, keepdim=True)])
        a, b, c = f.unbind(1)
        f = torch.stack([torch.stack(t, 1) for t in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))],
                        1).reshape(-1, 3)
    return (v @ _turn(g).T).float().contiguous(), f.int().contiguous()


def _terrain(cells, g):
    """Height field on [-1, 1]^2: four octaves of value noise of amplitude 0.2."""
    x = torch.linspace(-1.0, 1.0, cells + 1, dtype=torch.float64, device="cuda")
    h = torch.zeros(cells + 1, cells + 1, dtype=torch.float64, device="cuda")
    for o in range(4):
        m = 4 << o
        lattice = 2.0 * _rand(g, m + 2, m + 2) - 1.0
        at = (x + 1.0) * 0.5 * m
        i = at.floor().long().clamp(0, m - 1)
        s = at - i
        s = s * s * (3.0 - 2.0 * s)
        rows = lattice[i] + (lattice[i + 1] - lattice[i]) * s[:, None]
        h += 0.5 ** o * (rows[:, i] + (rows[:, i + 1] - rows[:, i]) * s[None, :])
    h *= 0.2 / 1.875
    z, xx = torch.meshgrid(x, x, indexing="ij")
    v = torch.stack([xx, h, z], -1).reshape(-1, 3).float().contiguous()
    j, i = torch.meshgrid(torch.arange(cells, device="cuda"), torch.arange(cells, device="cuda"), indexing="ij")
    a = (j * (cells + 1) + i).reshape(-1)
    b, c, d = a + 1, a + cells + 2, a + cells + 1
    f = torch.stack([torch.stack([a, c, b], 1), torch.stack([a, d, c], 1)], 1).reshape(-1, 3)
    return v, f.int().contiguous()


def _soup(n, g):
    """Triangles with edges log-uniform in [1e-3, 1e-1] around eight Gaussian clusters."""
    mean = -0.4 + 0.8 * _rand(g, 8, 3)
    sigma = 0.02 * 5.0 ** _rand(g, 8)
    weight = -torch.log1p(-_rand(g, 8))
    of = torch.bucketize(_rand(g, n), (weight / weight.sum()).cumsum(0)).clamp_max(7)
    c = mean[of] + sigma[of, None] * torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    edge = 1e-3 * 100.0 ** _rand(g, n)
    a = _unit(g, n)
    helper = torch.zeros_like(a)
    helper[torch.arange(n, device="cuda"), (a[:, 0].abs() >= 0.9).long()] = 1.0
    b1 = torch.linalg.cross(a, helper)
    b1 = b1 / b1.norm(dim=1, keepdim=True)
    b2 = torch.linalg.cross(a, b1)
    turn = 2.0 * math.pi * (_rand(g, n)[:, None] + torch.arange(3, device="cuda") / 3.0)
    v = c[:, None] + (edge / math.sqrt(3.0))[:, None, None] * (turn.cos()[..., None] * b1[:, None] +
                                                               turn.sin()[..., None] * b2[:, None])
    return (v.reshape(-1, 3).float().contiguous(),
            torch.arange(3 * n, dtype=torch.int32, device="cuda").reshape(n, 3))


def _spheres(n, g):
    """Centres in [-50, 50]^3, radii log-uniform in [0.01, 1]; boxes a little outside them."""
    s = torch.cat([100.0 * _rand(g, n, 3) - 50.0, 0.01 * 100.0 ** _rand(g, n, 1)], 1).float()
    r = s[:, 3:].double() * (1.0 + 1e-6) + 1e-5
    return s.contiguous(), torch.cat([s[:, :3] - r, s[:, :3] + r], 1).float().contiguous()


def _camera_rays(eye, width, height):
    """Pinhole rays through the pixel centres, looking down -z, 60 degrees high."""
    th = math.tan(math.radians(30.0))
    x = (2.0 * (torch.arange(width, dtype=torch.float64, device="cuda") + 0.5) / width - 1.0) * th * width / height
    y = (1.0 - 2.0 * (torch.arange(height, dtype=torch.float64, device="cuda") + 0.5) / height) * th
    d = torch.stack([x[None].expand(height, width), y[:, None].expand(height, width),
                     torch.full((height, width), -1.0, dtype=torch.float64, device="cuda")], -1).reshape(-1, 3)
    return _rays(torch.as_tensor(eye, device="cuda").expand_as(d), d / d.norm(dim=1, keepdim=True))


def _rays(o, d):
    n = o.shape[0]
    zero = torch.zeros(n, 1, dtype=torch.float64, device="cuda")
    return torch.cat([o, zero, d, zero + math.inf], 1).float().contiguous()


def _random_rays(n, lo, hi, g):
    return _rays(lo + (hi - lo) * _rand(g, n, 3), _unit(g, n))


def _frames(n, g):
    """Rotations x y z w, scales in [0.5, 2], translations in [-10, 10]^3."""
    return torch.cat([_quaternions(g, n), 0.5 + 1.5 * _rand(g, n, 3), 20.0 * _rand(g, n, 3) - 10.0],
                     1).float().contiguous()


def _mesh(case, seed):
    g = _rng(seed, 1)
    return {"icosphere": _icosphere, "terrain": _terrain, "soup": _soup}[case["shape"]](case["size"], g)


def _world(vertices, frames):
    """World vertices (instances, vertices, 3) in 64 bits."""
    f = frames.double()
    return (vertices.double()[None] * f[:, None, 4:7]) @ _matrix(f[:, :4]).transpose(1, 2) + f[:, None, 7:10]


def _scene_inputs(case, seed):
    """Mesh, instance frames, camera rays and extent of an instanced scene."""
    v, f = _mesh(case, seed)
    frames = _frames(case["instances"], _rng(seed, 2))
    w = _world(v, frames)
    lo, hi = w.amin((0, 1)), w.amax((0, 1))
    extent = float((hi - lo).max())
    eye = 0.5 * (lo + hi)
    eye[2] += case["distance"] * extent
    return v, f, frames, _camera_rays(eye, case["width"], case["height"]), extent


def _mesh_rays(case, seed):
    """Mesh and camera rays of a single geometry."""
    v, f = _mesh(case, seed)
    return v, f, _camera_rays([0.0, 0.0, case["distance"]], case["width"], case["height"])


# ---------------------------------------------------------------- what a program keeps
class _State:
    """Tensors and library objects of one case, by name."""

    def __init__(self, **kept):
        self.__dict__.update(kept)


class _Owner:
    """Library objects that are given back, in this order, when nothing refers to them any more."""

    def __init__(self, *kept):
        self.kept = kept

    def __del__(self):
        for x in self.kept:
            x.close()


class _Words:
    """32-bit words of device memory that belong to a library object, which they keep alive."""

    def __init__(self, at, rows, width, owner):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (rows, width), "typestr": "<i4", "data": (int(at), False),
                                         "version": 3, "strides": None}


def _flags(case):
    return grt.GRT_BUILD_PREFER_FAST | (grt.GRT_BUILD_WIDE8_NODES if case.get("wide8") else 0)


def _views(geometry, shape, owner):
    """The buffers a build fills, as they lie in the library."""
    i = geometry.info()
    leaf = 1 if shape == "spheres" else 12

    def words(at, rows, width):
        return torch.as_tensor(_Words(at, rows, width, owner), device="cuda")

    out = {"nodes": words(i.nodes, i.nodeCount, 16), "wide": words(i.wideNodes, i.nodeCount, 32)[:, :28],
           "leaves": words(i.leaves, i.leafCount, leaf), "parents": words(i.parents, 2 * i.leafCount - 1, 1)}
    if i.wide8Nodes:
        out["wide8"] = words(i.wide8Nodes, i.nodeCount, 64)
    return out


def prepare(case, seed):
    ctx, kind, flags = _ctx(), case["kind"], _flags(case)
    if kind == "build":
        if case["shape"] == "spheres":
            spheres, boxes = _spheres(case["size"], _rng(seed, 1))
            geometry = objects.Geometry(ctx, boxes=boxes, build_flags=flags)
        else:
            v, f = _mesh(case, seed)
            geometry = objects.Geometry(ctx, vertices=v, indices=f, build_flags=flags)
        owner = _Owner(geometry)
        geometry.build()
        return _State(kind=kind, geometry=geometry, views=_views(geometry, case["shape"], owner))
    if kind == "lambert":
        v, f, rays, colours, light, target = _lambert_inputs(case, seed)
        geometry = objects.Geometry(ctx, vertices=v, indices=f).build()
        renderer = shading.LambertRenderer(ctx, geometry, f, rays, store=case["store"])
        leaves = [x.clone().requires_grad_() for x in (colours, light, v)]
        return _State(kind=kind, owner=_Owner(geometry), renderer=renderer, leaves=leaves, target=target)
    if kind == "batch":
        geometries, scenes, hits = [], [], [None] * case["scenes"]
        for k, v, f, rays in _batch_inputs(case, seed):
            geometries.append(objects.Geometry(ctx, vertices=v, indices=f))
            hits[k] = objects.new_hits(rays.shape[0])
            scenes.append((geometries[-1], rays, hits[k]))
        batch = objects.Batch(ctx, scenes, grt.batch_options(graph=True))
        return _State(kind=kind, owner=_Owner(batch, *geometries), batch=batch, hits=hits)
    if case["shape"] == "spheres":
        spheres, boxes = _spheres(case["size"], _rng(seed, 1))
        half = torch.full((3,), 50.0, dtype=torch.float64, device="cuda")
        rays = _random_rays(case["rays"], -half, half, _rng(seed, 2))
        geometry = objects.Geometry(ctx, boxes=boxes, build_flags=flags).build()
        table = objects.FuncTable(ctx)
        table.set(0, 0, grt.GRT_INTERSECT_SPHERE, spheres)
        return _State(kind="spheres", owner=_Owner(geometry, table), geometry=geometry, table=table, rays=rays,
                      hits=objects.new_hits(rays.shape[0]), any=objects.new_hits(rays.shape[0]))
    if not case["instances"]:
        v, f, rays = _mesh_rays(case, seed)
        geometry = objects.Geometry(ctx, vertices=v, indices=f, build_flags=flags).build()
        return _State(kind=kind, owner=_Owner(geometry), geometry=geometry, scene=None, rays=rays,
                      hits=objects.new_hits(rays.shape[0]))
    v, f, frames, rays, extent = _scene_inputs(case, seed)
    geometry = objects.Geometry(ctx, vertices=v, indices=f, build_flags=flags).build()
    scene = objects.Scene(ctx, [geometry.handle] * case["instances"], frames, build_flags=flags).build()
    hits = objects.new_hits(rays.shape[0])
    state = _State(kind=kind, owner=_Owner(scene, geometry), scene=scene, rays=rays, hits=hits)
    if kind == "ao":
        grt.grtTraceClosest(ctx.handle, scene.handle, None, rays, rays.shape[0], hits)
        state.samples, state.length, state.seed = case["samples"], 0.05 * extent, int(seed)
        state.ao = torch.empty(rays.shape[0], device="cuda")
    return state


def _lambert_inputs(case, seed):
    """Mesh, camera rays, per-vertex colours, light direction and a target image."""
    g = _rng(seed, 3)
    v, f = _icosphere(case["size"], _rng(seed, 1))
    rays = _camera_rays([0.0, 0.0, 3.0], case["width"], case["height"])
    light = torch.ones(3, dtype=torch.float64, device="cuda") / math.sqrt(3.0) + 0.1 * _unit(g, 1)[0]
    return (v, f, rays, _rand(g, v.shape[0], 3).float(), (light / light.norm()).float(),
            _rand(g, rays.shape[0], 3).float())


def _batch_sizes(case):
    """(triangles, rays) of each soup, both spread evenly over the logarithm of their range."""
    m = case["scenes"]
    return [(int(1000 * (case["most"] / 1000) ** ((k + 0.5) / m)),
             int(4096 * (case["most_rays"] / 4096) ** ((k * 11 % m + 0.5) / m))) for k in range(m)]


def _batch_inputs(case, seed):
    """The soups in an order of the seed's, half camera rays and half random rays for each."""
    g = _rng(seed, 4)
    sizes = _batch_sizes(case)
    for k in torch.argsort(_rand(g, len(sizes))).tolist():
        n, r = sizes[k]
        v, f = _soup(n, g)
        lo, hi, eye = v.amin(0).double(), v.amax(0).double(), v.double().mean(0)
        eye[2] += 1.5
        side = int(math.sqrt(r / 2))
        yield k, v, f, torch.cat([_camera_rays(eye, side, side), _random_rays(r - side * side, lo, hi, g)])


# ---------------------------------------------------------------- one pass
def _records(hits):
    return {"ids": hits[:, :2], "tuv": hits[:, 2:].view(torch.float32)}


def run(state):
    ctx = _ctx().handle
    if state.kind == "build":
        state.geometry.build()
        return state.views
    if state.kind == "batch":
        state.batch.run()
        return [_records(h) for h in state.hits]
    if state.kind == "lambert":
        colours, light, positions = state.leaves
        image = shading.lambert_shade(colours, light, positions, state.renderer)
        loss = (image - state.target).square().sum()
        return [image.detach(), *torch.autograd.grad(loss, state.leaves)]
    n = state.rays.shape[0]
    if state.kind == "ao":
        grt.grtTraceAmbientOcclusion(ctx, state.scene.handle, state.rays, state.hits, n, state.samples, state.seed,
                                     state.length, state.ao)
        return state.ao
    if state.kind == "spheres":
        grt.grtTraceClosest(ctx, None, state.geometry.handle, state.rays, n, state.hits, state.table.handle)
        grt.grtTraceAnyHit(ctx, None, state.geometry.handle, state.rays, n, state.any, state.table.handle)
        return [_records(state.hits), _records(state.any)]
    grt.grtTraceClosest(ctx, state.scene and state.scene.handle, None if state.scene else state.geometry.handle,
                        state.rays, n, state.hits)
    return _records(state.hits)


def _primitives(case):
    if case["kind"] == "lambert" or case["shape"] == "icosphere":
        return 20 * 4 ** case["size"]
    return 2 * case["size"] ** 2 if case["shape"] == "terrain" else case["size"]


def _trace_work(rays, primitives):
    """Each ray in and its record out, the tree and the primitives once; per ray the boxes
    of a walk to one leaf of a 4-wide tree (12 operations each) and one primitive test."""
    levels = max(1.0, math.log(primitives, 4))
    return {"bytes": 52 * rays + 112 * primitives, "flops": rays * (48 * levels + 60)}


def _build_work(n, mesh, wide8=False):
    """Primitives in; binary and 4-wide nodes, leaves, links (and 8-wide nodes) out."""
    return {"bytes": n * ((48 if mesh else 24) + 64 + 112 + (52 if mesh else 4) + 8 + (256 if wide8 else 0)),
            "flops": 100 * n}


def work(case):
    kind = case["kind"]
    if kind == "build":
        return _build_work(_primitives(case), case["shape"] != "spheres", case["wide8"])
    if kind == "batch":
        total = {"bytes": 0, "flops": 0}
        for n, r in _batch_sizes(case):
            for w in (_build_work(n, True), _trace_work(r, n)):
                total = {key: total[key] + w[key] for key in total}
        return total
    rays = case["rays"] if "rays" in case else case["width"] * case["height"]
    w = _trace_work(rays, _primitives(case))
    if kind == "lambert":  # forward as above; image, target and its gradient; records read back
        return {"bytes": w["bytes"] + rays * (12 * 4 + 52), "flops": w["flops"] + 200 * rays}
    if kind == "ao":  # the records in and one value out; the shadow rays themselves stay on chip
        return {"bytes": 56 * rays + 112 * _primitives(case), "flops": 0.06 * case["samples"] * w["flops"]}
    if case["shape"] == "spheres":  # closest and any hit
        return {"bytes": w["bytes"] + 52 * rays, "flops": 2 * w["flops"]}
    return w


# ---------------------------------------------------------------- in 64 bits
def _plucker(o, d, tri, best, ids, base):
    """Nearest crossing of rays (o, d) with triangles tri (n, 3, 3), folded into best and ids."""
    a, e1, e2 = tri[:, 0], tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
    n = torch.linalg.cross(e1, e2)
    m = torch.linalg.cross(o, d)
    for at in range(0, o.shape[0], max(1, (1 << 27) // max(1, tri.shape[0]))):
        s = slice(at, at + max(1, (1 << 27) // max(1, tri.shape[0])))
        det = -(d[s] @ n.T)
        # Moller-Trumbore's triple products as products of matrices
        u = (m[s] @ e2.T + d[s] @ torch.linalg.cross(a, e2).T) / det
        v = -(m[s] @ e1.T + d[s] @ torch.linalg.cross(a, e1).T) / det
        t = (o[s] @ n.T - (a * n).sum(1)) / det
        t = torch.where((det != 0) & (u >= 0) & (v >= 0) & (u + v <= 1) & (t >= 0), t, math.inf)
        near, which = t.min(1)
        old = best[s]
        ids[s] = torch.where(near < old, which + base, ids[s])
        best[s] = torch.minimum(near, old)


def _barycentrics(o, d, a, b, c):
    """t, u, v of rays on the planes of their triangles."""
    e1, e2, w = b - a, c - a, o - a
    p, q = torch.linalg.cross(d, e2), torch.linalg.cross(w, e1)
    det = (e1 * p).sum(1)
    return (e2 * q).sum(1) / det, (w * p).sum(1) / det, (d * q).sum(1) / det


def _closest64(o, d, tri):
    best = torch.full((o.shape[0],), math.inf, dtype=torch.float64, device="cuda")
    ids = torch.full((o.shape[0],), -1, dtype=torch.int64, device="cuda")
    _plucker(o, d, tri, best, ids, 0)
    return best, ids


def _tuv64(o, d, tri, best, ids):
    hit = ids >= 0
    out = torch.zeros(o.shape[0], 3, dtype=torch.float64, device="cuda")
    out[:, 0] = math.inf
    k = tri[ids[hit]]
    out[hit] = torch.stack(_barycentrics(o[hit], d[hit], k[:, 0], k[:, 1], k[:, 2]), 1)
    return out


def _scene64(case, seed):
    """Closest hits through all instances: each ray against the tiles of triangles (512 at
    a time) whose boxes it meets in object space."""
    v, f, frames, rays, _ = _scene_inputs(case, seed)
    o, d = rays[:, :3].double(), rays[:, 4:7].double()
    g = frames.double()
    turn = _matrix(g[:, :4])
    cells, step = case["size"], 16
    t4 = torch.nn.functional.pad(f.long().reshape(cells, cells, 2, 3), (0, 0, 0, 0, 0, -cells % step, 0, -cells % step),
                                 value=-1)
    m = t4.shape[0] // step
    tiles = t4.reshape(m, step, m, step, 2, 3).transpose(1, 2).reshape(m * m, -1, 3)
    p = v.double()
    best = torch.full((o.shape[0],), math.inf, dtype=torch.float64, device="cuda")
    out = torch.zeros(o.shape[0], 3, dtype=torch.float64, device="cuda")
    boxes = []
    for tile in tiles:
        k = p[tile[tile[:, 0] >= 0]]
        boxes.append((k, k.amin((0, 1)) - 1e-9, k.amax((0, 1)) + 1e-9))
    lo, hi = p.amin(0) - 1e-9, p.amax(0) + 1e-9
    for i in range(g.shape[0]):
        oo = (o - g[i, 7:10]) @ turn[i] / g[i, 4:7]
        dd = d @ turn[i] / g[i, 4:7]

        def meets(ro, rd, a, b):
            x, y = (a - ro) / rd, (b - ro) / rd
            return torch.minimum(x, y).amax(1).clamp_min(0) <= torch.maximum(x, y).amin(1)

        some = meets(oo, dd, lo, hi).nonzero()[:, 0]
        so, sd = oo[some], dd[some]
        for k, a, b in boxes:
            at = meets(so, sd, a, b).nonzero()[:, 0]
            if not at.numel():
                continue
            centre = 0.5 * (a + b)
            ro, rd = so[at] - centre, sd[at]
            near, which = _closest64(ro, rd, k - centre)
            won = (near < best[some[at]]).nonzero()[:, 0]
            to, c = some[at[won]], (k - centre)[which[won]]
            tuv = torch.stack(_barycentrics(ro[won], rd[won], c[:, 0], c[:, 1], c[:, 2]), 1)
            best[to], out[to] = tuv[:, 0], tuv
    out[:, 0] = best
    return out


def _lambert64(case, seed):
    v, f, rays, colours, light, target = _lambert_inputs(case, seed)
    o, d = rays[:, :3].double(), rays[:, 4:7].double()
    c, l, p = (x.double().requires_grad_() for x in (colours, light, v))
    best, ids = _closest64(o, d, p.detach()[f.long()])
    hit = (ids >= 0).nonzero()[:, 0]
    k = f.long()[ids[hit]]
    a, b, e = p[k[:, 0]], p[k[:, 1]], p[k[:, 2]]
    t, u, w = _barycentrics(o[hit], d[hit], a, b, e)
    n = torch.linalg.cross(b - a, e - a)
    n = n / n.norm(dim=1, keepdim=True)
    n = torch.where(((n * d[hit]).sum(1) > 0)[:, None], -n, n)
    facing = (n * l).sum(1)
    start = (o[hit] + d[hit] * t[:, None] + 1e-4 * n).detach()
    dark, _ = _closest64(start, l.detach().expand_as(start).contiguous(), p.detach()[f.long()])
    lit = (facing > 0) & dark.isinf()
    colour = (1 - u - w)[:, None] * c[k[:, 0]] + u[:, None] * c[k[:, 1]] + w[:, None] * c[k[:, 2]]
    image = torch.zeros(o.shape[0], 3, dtype=torch.float64, device="cuda")
    image = image.index_put((hit,), torch.where(lit, facing, 0.0)[:, None] * colour)
    grads = torch.autograd.grad((image - target.double()).square().sum(), (c, l, p))
    return [image.detach(), *grads]


def exact(case, seed):
    """Hit distances and barycentrics, images and gradients in 64 bits. Builds move words
    and take minima; occlusion counts samples; the hits of a million spheres and of many
    soups take too long without a tree."""
    if case["kind"] == "lambert":
        return _lambert64(case, seed)
    if case["kind"] != "trace" or case["shape"] == "spheres":
        return None
    if case["instances"]:
        return {"ids": None, "tuv": _scene64(case, seed)}
    v, f, rays = _mesh_rays(case, seed)
    o, d, tri = rays[:, :3].double(), rays[:, 4:7].double(), v.double()[f.long()]
    return {"ids": None, "tuv": _tuv64(o, d, tri, *_closest64(o, d, tri))}
