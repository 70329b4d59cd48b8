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

    def get(self, attr, pool=None):
        v = ctypes.c_uint64()
        self.ok(self.cu.cuMemPoolGetAttribute(pool or self.default, attr, ctypes.byref(v)))
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
        torch.cuda.synchronize()
        assert self.get(USED_CURRENT, pool) == 0  # whatever f() took is given back
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


@pytest.mark.parametrize("n_rhs", [0, 3])
def test_coarsest_inverse_in_place(n_rhs):
    """A hierarchy of one level of 5,202 unknowns: setup needs the 216 MB of its inverse and little else (K takes
    8 MB), in the V-cycles of both precisions and in the batch."""
    tam = need_gpu()
    pools = Pools()
    pb = meshgen.slab_box_problem(16, 16, 5)
    d = tam.problem_to_device(pb)
    K, rhs = tam.fem_assemble_elasticity(**d)
    prm = tam.amg_params_default(coarse_max_dofs=6000, level_precision=1 if n_rhs else 0)
    N = 3 * pb.n_nodes
    hs = []
    peak = pools.peak(lambda: hs.append(tam.amg_setup(K, d["coords"], prm)))
    H = hs[0]
    assert tam.amg_info(H)["n_levels"] == 1 and N > 5000
    assert 8 * N * N <= peak <= 1.25 * 8 * N * N
    free = d["dirichlet_mask"] == 0
    r = torch.randn((pb.n_nodes, 3), dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    r[~free] = 0.0
    if n_rhs:
        B = torch.stack([r.reshape(-1) * (k + 1) for k in range(n_rhs)])
        X = torch.zeros_like(B)
        its, _, _ = tam.amg_pcg_solve_batch([H], [B], [X], rtol=1e-10)
        assert max(its) <= 2
        z = (X[-1] / n_rhs).reshape(r.shape)
    else:
        z = tam.amg_vcycle(H, r)
    assert tam.tam_matrix_residual_norm(K, r, z) <= 1e-8 * float(r.norm())


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_batch_after_running_out_of_memory(precision):
    """A batched solve that runs out of memory, at any stage of building its operators and workspace, says so and
    gives back what it took; a later call with enough memory gives the solutions of a hierarchy that never did."""
    tam = need_gpu()
    pools = Pools()
    pb = meshgen.slab_box_problem(96, 24, 24)
    d = tam.problem_to_device(pb)
    K, rhs = tam.fem_assemble_elasticity(**d)
    prm = tam.amg_params_default(level_precision=precision)
    B = torch.stack([rhs.reshape(-1) * (k + 1) for k in range(8)])

    def solve(H):
        X = torch.zeros_like(B)
        tam.amg_pcg_solve_batch([H], [B], [X], rtol=1e-8)
        return X

    fresh = tam.amg_setup(K, d["coords"], prm)
    ref = []
    peak = pools.peak(lambda: ref.append(solve(fresh)))
    fresh.destroy()
    H = tam.amg_setup(K, d["coords"], prm)

    def short():
        with pytest.raises(tam.TamError) as e:
            solve(H)
            pytest.skip("the driver does not limit the pool")
        assert e.value.code == -3, e.value  # TAM_ERR_OOM

    for part in (0.05, 0.2, 0.35, 0.5, 0.65, 0.8):
        pools.limited(int(part * peak), short)
    X = solve(H)
    assert float((X - ref[0]).norm()) <= 1e-6 * float(ref[0].norm())


def test_batch_operators_are_not_kept_twice():
    """The batched solve on an FP64 hierarchy keeps one FP32 copy of every operator.  Copies and workspace are those
    of an FP32 hierarchy and its own batch, less the latter's second copies of the operators whose solves read a
    lanes-per-row store (at least 100 MB on this machine, whose first restriction is one)."""
    tam = need_gpu()
    pools = Pools()
    pb = meshgen.slab_box_problem(256, 64, 64)
    d = tam.problem_to_device(pb)
    K, rhs = tam.fem_assemble_elasticity(**d)
    B = torch.stack([rhs.reshape(-1)] * 2)

    def batch(H):
        X = torch.zeros_like(B)
        tam.amg_pcg_solve_batch([H], [B], [X], rtol=1e-8, max_iter=2, raise_on_error=False)

    kept, extra = [], []
    for precision in (0, 1):
        before = pools.get(USED_CURRENT)
        H = tam.amg_setup(K, d["coords"], tam.amg_params_default(level_precision=precision))
        kept.append(pools.get(USED_CURRENT) - before)
        extra.append(pools.peak(lambda: batch(H)))
        twice = 0
        for l in range(tam.amg_info(H)["n_levels"] - 1):
            for which in range(3):  # A, P, R
                if tam.amg_level_spmv_plan(H, l, which)["kind"] == 1:
                    e = tam.amg_level_export(H, l, which)
                    twice += 4 * e["nnzb"] * e["br"] * e["bc"]
        H.destroy()
    assert twice > 100e6
    assert extra[0] <= kept[1] - kept[0] + extra[1] - 0.9 * twice
