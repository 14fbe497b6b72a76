"""Device memory an operation holds at its peak: no more than with one allocation per temporary and one rotation or giant step
at a time, and several rotations at once give way to one at a time where the memory is short."""
import ctypes

import numpy as np
import pytest

from paper_2606_10477_gb300 import hedap, inputs

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, CU_MEMPOOL_ATTR_USED_MEM_HIGH


class _Location(ctypes.Structure):
    _fields_ = [("type", ctypes.c_int), ("id", ctypes.c_int)]


class _PoolProps(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location", _Location),
                ("win32", ctypes.c_void_p), ("max_size", ctypes.c_size_t), ("usage", ctypes.c_ushort),
                ("reserved", ctypes.c_ubyte * 54)]


class Pools:
    def __init__(self):
        import torch
        torch.zeros(1, device="cuda")
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.dev = ctypes.c_int()
        assert self.cu.cuCtxGetDevice(ctypes.byref(self.dev)) == 0
        self.default = ctypes.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.default), self.dev) == 0

    def used(self, attr):
        v = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.default, attr, ctypes.byref(v)) == 0
        return v.value

    def peak(self, call, ctx):
        """Bytes above what is held before, at the peak of a second call (the first one builds the tables and keys)."""
        call()
        ctx.sync()
        assert self.cu.cuMemPoolSetAttribute(self.default, USED_HIGH, ctypes.byref(ctypes.c_uint64(0))) == 0
        before = self.used(USED_CURRENT)
        out = call()
        ctx.sync()
        high = self.used(USED_HIGH) - before
        del out
        return high

    def limited(self, max_size):
        props = _PoolProps(alloc_type=1, location=_Location(1, self.dev.value), max_size=max_size)  # pinned, on the device
        pool = ctypes.c_void_p()
        assert self.cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
        return pool


@pytest.mark.parametrize("log_n", [10, 14])
@pytest.mark.parametrize("n_q,n_p,alpha,level", [(12, 1, 1, 11), (8, 2, 2, 3), (12, 4, 4, 11), (8, 2, 2, 1)])
@pytest.mark.parametrize("batch", [1, 5])
def test_peak_of_products_and_rotations(log_n, n_q, n_p, alpha, level, batch):
    g = hedap.Context(log_n, [50] * n_q, [60] * n_p, alpha, 40.0, 64, 1)
    x = [inputs.random_ciphertext_limbs(3 + k, g.primes(), level, g.N) for k in range(batch)]
    a = g.pack([g.ct_import(v, level, g.scale) for v in x])
    unit = 8 * batch * g.N
    ct, ext, dn = 2 * (level + 1), level + 1 + n_p, -(-(level + 1) // alpha)
    switch = 2 * ext + max(ct // 2 + dn * ext, ct)  # sums, then the ModUp's limbs and digits or ModDown's limbs
    p = Pools()
    slack = 1 << 14
    assert p.peak(lambda: g.mul(a, a), g) <= unit * max(ct + ct // 2 + 2 * ext + ct // 2 + dn * ext,
                                                       ct + 2 * ext + 2 * level + 4 + 2 * level) + slack
    assert p.peak(lambda: g.mul_relin(a, a), g) <= unit * (ct + ct // 2 + switch) + slack
    assert p.peak(lambda: g.rotate(a, 1), g) <= unit * (ct + switch) + slack


@pytest.mark.parametrize("groups", [1, 2])
@pytest.mark.parametrize("inverse", [True, False])
def test_peak_of_a_linear_transform(groups, inverse):
    """The baby steps, one giant step's sum, its ModDown, the result so far, and the rotation's result and workspace."""
    g = hedap.Context(10, [45] + [36] * 8, [50, 50], 2, 36.0, 0, 1)
    g.bts_setup(K=28, r=0, deg=2, cts=groups, stc=groups)
    level = g.n_q - 1
    c = g.encrypt(inputs.uniform_values(7, g.N // 2, -1, 1), level, 9)
    ct, ext, dn = 2 * (level + 1), level + 1 + g.n_p, -(-(level + 1) // g.alpha)
    rotation = ct + 2 * ext + ct // 2 + dn * ext
    bound = 8 * g.N * (16 * 2 * ext + 2 * ext + ct + ct + rotation)
    assert Pools().peak(lambda: g.linear_transform_group(c, groups, inverse, 0, c.scale / 16), g) <= bound


def test_hoisted_rotations_in_short_memory():
    """16 rotations of a batch whose sums and workspaces do not fit at once: the words of an unlimited run."""
    g = hedap.Context(14, [50] * 8, [60, 60], 2, 50.0, 64, 1)
    level, batch, steps = 7, 8, list(range(1, 17))
    a = g.pack([g.ct_import(inputs.random_ciphertext_limbs(60 + k, g.primes(), level, g.N), level, g.scale)
                for k in range(batch)])
    want = [c.limbs() for r in g.rotate_hoisted(a, steps) for c in (g.unpack(r, 0), g.unpack(r, batch - 1))]
    g.sync()
    mb = 8 * batch * g.N / 1e6
    ext, ct = 10, 16
    one = mb * (4 * ext + 2 * ext + ct + 16 * ct)  # digits, sums, ModDown, results
    all_ = mb * (4 * ext + 16 * (2 * ext + ct + ct))
    limit = int(0.5 * (one + all_))
    assert one + 64 < limit < all_ - 64
    p = Pools()
    pool = p.limited(limit << 20)
    assert p.cu.cuDeviceSetMemPool(p.dev, pool) == 0
    try:
        rot = g.rotate_hoisted(a, steps)
        g.sync()
    finally:
        assert p.cu.cuDeviceSetMemPool(p.dev, p.default) == 0
    got = [c.limbs() for r in rot for c in (g.unpack(r, 0), g.unpack(r, batch - 1))]
    assert all(np.array_equal(x, y) for x, y in zip(got, want))
    del rot
    g.sync()
    assert p.cu.cuMemPoolDestroy(pool) == 0


def test_context_of_a_small_ring_in_short_memory():
    """The tuner's scratch for a small ring's large batches (16 MiB) is not needed: with room for the rest only (17 of 32 MiB),
    the context is made, and its products are those of any other."""
    p = Pools()
    pool = p.limited(32 << 20)
    assert p.cu.cuDeviceSetMemPool(p.dev, pool) == 0
    try:
        g = hedap.Context(13, [45] * 4, [60], 1, 40.0, 64, 1)
        x = inputs.random_ciphertext_limbs(5, g.primes(), 3, g.N)
        got = g.mul(g.ct_import(x, 3, g.scale), g.ct_import(x, 3, g.scale)).limbs()
        g.sync()
        g.close()
    finally:
        assert p.cu.cuDeviceSetMemPool(p.dev, p.default) == 0
    h = hedap.Context(13, [45] * 4, [60], 1, 40.0, 64, 1)
    assert np.array_equal(got, h.mul(h.ct_import(x, 3, h.scale), h.ct_import(x, 3, h.scale)).limbs())
