"""Sorts by any number of significant bits, odd and even numbers of passes, from one key to the
edges of one tile and beyond, equal a stable numpy sort by those bits; the scratch is any memory."""
import numpy as np
import pytest
import torch

import paper_2603_00292_gb300 as grt
from paper_2603_00292_gb300.objects import device_tensor, empty_bytes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 100, 1024, 1025, 2047, 2048, 2049, 5000, 300_001])
@pytest.mark.parametrize("key_bits, bits", [(32, 1), (32, 8), (32, 9), (32, 17), (32, 24), (32, 32), (64, 8), (64, 33),
                                            (64, 56), (64, 64)])
def test_significant_bits(gpu, n, key_bits, bits):
    rng = np.random.default_rng([n, bits])
    kd = np.uint32 if key_bits == 32 else np.uint64
    keys = (rng.integers(0, 1 << 63, n, dtype=np.uint64) & np.uint64((1 << bits) - 1)).astype(kd)
    k, v = device_tensor(keys), device_tensor(np.arange(n, dtype=np.int32)[::-1].copy())
    temp = empty_bytes(grt.grtSortTemporaryBufferSize(n, key_bits))
    temp.fill_(0xC7)
    for _ in range(2):  # the second on sorted keys and the first one's leavings
        grt.grtSortPairs(gpu.handle, k, v, n, key_bits, bits, temp)
    torch.cuda.synchronize()
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(k.cpu().numpy().view(kd), keys[order])
    assert np.array_equal(v.cpu().numpy(), (n - 1 - order).astype(np.int32))
    assert grt.grtGetLastDeviceError(gpu.handle) == grt.GRT_SUCCESS
