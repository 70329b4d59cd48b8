"""Device memory that a call needs at its peak, from the stream-ordered pool's counters and under a limit."""
import ctypes

import pytest

from gpu_util import need_gpu, torch
from paper_1804_10060_gb300 import meshgen

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_*


class PoolProps(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("win32", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


class Pools:
    def __init__(self):
        torch.zeros(1, device="cuda")
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.default = ctypes.c_void_p()
        self.ok(self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.default), 0))

    def ok(self, r):
        assert r == 0, r

    def get(self, attr):
        v = ctypes.c_uint64()
        self.ok(self.cu.cuMemPoolGetAttribute(self.default, attr, ctypes.byref(v)))
        return v.value

    def peak(self, f):
        """Bytes beyond those in use that f() needs at its peak."""
        torch.cuda.synchronize()
        self.ok(self.cu.cuMemPoolSetAttribute(self.default, USED_HIGH, ctypes.byref(ctypes.c_uint64(0))))
        before = self.get(USED_CURRENT)
        f()
        torch.cuda.synchronize()
        return self.get(USED_HIGH) - before

    def limited(self, size, f):
        """f() with a pool of its own of at most `size` bytes."""
        pool, p = ctypes.c_void_p(), PoolProps(alloc_type=1, location_type=1, location_id=0, max_size=size)
        self.ok(self.cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(p)))
        self.ok(self.cu.cuDeviceSetMemPool(0, pool))
        try:
            f()
            torch.cuda.synchronize()
        finally:
            self.ok(self.cu.cuDeviceSetMemPool(0, self.default))
            self.ok(self.cu.cuMemPoolDestroy(pool))


def test_matrix_outside_the_range_needs_no_split_copy():
    """A K outside the double-float range is kept without its split copy, so it also assembles where memory does not
    reach for one; a K inside the range is out of memory there."""
    tam = need_gpu()
    pools = Pools()
    pb = meshgen.slab_box_problem(80, 20, 20, degree=2)
    d = tam.problem_to_device(pb)
    far = dict(d, mat_props=d["mat_props"] * torch.tensor([2.0 ** 120, 1.0, 1.0], dtype=torch.float64, device="cuda"))

    def assemble(q):
        K, _ = tam.fem_assemble_elasticity(**q)
        y = tam.tam_matrix_spmv(K, d["coords"])
        n, nnzb, _ = K.info()
        K.destroy()
        return y, nnzb

    y, nnzb = assemble(far)
    peak = pools.peak(lambda: assemble(d))
    limit = peak - 36 * nnzb  # half a split copy (8 bytes for each of a block's 9 values) too little

    def short():
        with pytest.raises(tam.TamError) as e:
            assemble(d)
            pytest.skip("the driver does not limit the pool")
        assert e.value.code == -3, e.value  # TAM_ERR_OOM
        ys, _ = assemble(far)
        assert float((ys - y).norm()) <= 1e-13 * float(y.norm())

    pools.limited(limit, short)
    pools.limited(peak + (1 << 28), lambda: assemble(d))
