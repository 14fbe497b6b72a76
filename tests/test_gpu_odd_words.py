"""Transforms of device limbs that begin at an odd word run in place: no staging buffer, and the words of an aligned array."""
import ctypes

import numpy as np
import pytest

from paper_2606_10477_gb300 import hedap, inputs

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, CU_MEMPOOL_ATTR_USED_MEM_HIGH


def _pool():
    cu = ctypes.CDLL("libcuda.so.1")
    dev, pool = ctypes.c_int(), ctypes.c_void_p()
    assert cu.cuCtxGetDevice(ctypes.byref(dev)) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0

    def get(attr):
        v = ctypes.c_uint64()
        assert cu.cuMemPoolGetAttribute(pool, attr, ctypes.byref(v)) == 0
        return v.value

    def reset_high():
        assert cu.cuMemPoolSetAttribute(pool, USED_HIGH, ctypes.byref(ctypes.c_uint64(0))) == 0
    return get, reset_high


@pytest.mark.parametrize("log_n", [10, 12, 13, 14, 15, 17])
@pytest.mark.parametrize("inverse", [False, True])
def test_odd_words_in_place(log_n, inverse):
    import torch
    g = hedap.Context(log_n, [33, 45, 60], [60], 1, 30.0, 0, 1)
    primes = g.primes()
    polys = 2
    x = torch.from_numpy(inputs.random_limbs(3, np.tile(primes, polys), g.N).astype(np.int64)).cuda()
    want = g.ntt_batch(x.clone(), len(primes), 0, inverse=inverse)
    buf = torch.full((x.numel() + 2,), -1, dtype=torch.int64, device="cuda")
    odd = buf[1:-1].view(x.shape)
    odd.copy_(x)
    assert odd.data_ptr() % 16 == 8
    torch.cuda.synchronize()
    g.sync()
    get, reset_high = _pool()
    reset_high()
    before = get(USED_CURRENT)
    g.ntt_batch(odd, len(primes), 0, inverse=inverse)
    g.sync()
    assert get(USED_HIGH) <= before, "the transform allocated"
    assert torch.equal(odd, want) and buf[0] == -1 and buf[-1] == -1
