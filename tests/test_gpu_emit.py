"""Emission and fit of the linear BVH in blocks of 512 leaves and lists of 16 blocks, at the
edges of both, on trees that cross them in every way; the radix sort at its tiles' (2,048
keys) and groups' (8 tiles) edges. Everything is compared bit for bit with the oracle, or with
a stable numpy sort."""
import numpy as np
import pytest
import torch

import paper_2603_00292_gb300 as grt
from paper_2603_00292_gb300.objects import Geometry, device_tensor, empty_bytes
from test_gpu_build import check_bit_exact

pytestmark = pytest.mark.gpu


def _boxes(shape: str, n: int) -> np.ndarray:
    rng = np.random.default_rng(n)
    if shape == "random":
        c = rng.uniform(-1, 1, (n, 3))
    elif shape == "same":  # one code: the positions alone make the tree
        c = np.zeros((n, 3))
    elif shape == "runs":  # a few codes, each many times over
        c = rng.integers(0, 5, (n, 3)) * 0.25
    else:  # "comb": each next centroid half as far out, so subtrees hang off one long path
        c = np.zeros((n, 3))
        c[:, 0] = np.ldexp(1.0, -(np.arange(n) * 40 // n))
        c[:, 1] = rng.integers(0, 2, n) * c[:, 0]
    h = rng.uniform(0.0, 1e-3, (n, 3))
    return np.concatenate([c - h, c + h], axis=1).astype(np.float32)


@pytest.mark.parametrize("n", [2049, 4096, 4097, 8192, 8193, 8704, 131_072, 131_585])
@pytest.mark.parametrize("shape", ["random", "same", "runs", "comb"])
@pytest.mark.parametrize("bits", [30, 63])
def test_emission_at_block_edges(gpu, shape, n, bits):
    case = dict(boxes=_boxes(shape, n))
    g = Geometry(gpu, boxes=device_tensor(case["boxes"]), morton_bits=bits).build()
    check_bit_exact(g, case, bits)
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
    g.close()


@pytest.mark.parametrize("n", [2047, 2048, 2049, 16_384, 16_385, 34_816, 600_001])
@pytest.mark.parametrize("key_bits", [32, 64])
@pytest.mark.parametrize("kind", ["random", "equal", "high"])
def test_radix_sort_at_tile_edges(gpu, n, key_bits, kind):
    rng = np.random.default_rng(n)
    kd = np.uint32 if key_bits == 32 else np.uint64
    if kind == "random":
        keys = rng.integers(0, 1 << 62, n, dtype=np.uint64).astype(kd)
    elif kind == "equal":
        keys = np.full(n, 0xA5A5A5A5, dtype=kd)
    else:  # only the last digit differs
        keys = rng.integers(0, 256, n, dtype=np.uint64).astype(kd) << kd(key_bits - 8)
    k = device_tensor(keys)
    v = device_tensor(np.arange(n, dtype=np.int32)[::-1].copy())
    temp = empty_bytes(grt.grtSortTemporaryBufferSize(n, key_bits))
    grt.grtSortPairs(gpu.handle, k, v, n, key_bits, key_bits, temp)
    torch.cuda.synchronize()
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(k.cpu().numpy().view(kd), keys[order])
    assert np.array_equal(v.cpu().numpy(), (n - 1 - order).astype(np.int32))
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
