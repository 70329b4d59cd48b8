"""The tiled kernels at the sizes where a tile can go wrong: one item, a tile
less one, a tile, a tile and one, and a ragged last tile of several."""
import numpy as np
import pytest
import scipy.sparse as sp

from gpu_util import bsr_to_csr, need_gpu, sparse_rel, torch
from oracle import fem
from oracle import mlp as omlp
from oracle import thermal as oth
from paper_1804_10060_gb300 import meshgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells", [1, 31, 32, 33, 97])
@pytest.mark.parametrize("transient", [False, True])
def test_thermal_p2_cell_tiles(n_cells, transient):
    """Residual and Jacobian of n_cells quadratic cells of two materials (32 cells a block) against the
    oracle's exact integrals; FP64 sums of a few hundred terms: 1e-12 of the largest entry."""
    tam = need_gpu()
    pb = meshgen.unit_cube_problem(3, degree=2)
    cells = np.ascontiguousarray(pb.cells[:n_cells])
    used = np.unique(cells)
    back = -np.ones(pb.n_nodes, np.int64)
    back[used] = np.arange(used.size)
    n = used.size
    tp = meshgen.ThermalProblem(pb.coords[used], back[cells].astype(np.int32),
                                (np.arange(n_cells) % 2).astype(np.int32),
                                np.array([[1.5, 1.0, 5e-4, 0.05, 5e-5], [0.7, 2.0, 1e-3, 0.5, 2e-4]]),
                                np.zeros((0, 6), np.int32), np.zeros(0), np.zeros(n))
    d = tam.thermal_to_device(tp)
    th = tam.Thermal(d["coords"], d["cells"], d["cell_material"], tp.thermal_props, d["faces"])
    rng = np.random.default_rng(n_cells)
    T = 300.0 + 400.0 * rng.random(n)
    T_old = T - 20.0 * rng.random(n) if transient else None
    kw = dict(T_old=T_old, dt=0.05, theta=0.6) if transient else {}
    F = th.residual(torch.from_numpy(T).cuda(), torch.from_numpy(T_old).cuda() if transient else None,
                    kw.get("dt", 0.0), kw.get("theta", 1.0), d["beta"], d["T_bc"]).cpu().numpy()
    Fo, Jo = oth.assemble_thermal(tp, T, **kw)
    rp, ci, v = th.jacobian()
    J = sp.csr_matrix((v.cpu().numpy(), ci.cpu().numpy(), rp.cpu().numpy()), shape=(n, n))
    assert np.abs(F - Fo).max() <= 1e-12 * np.abs(Fo).max()
    assert abs(J - Jo).max() <= 1e-12 * abs(Jo).max()


@pytest.mark.parametrize("n_cells", [1, 31, 32, 33, 97])
@pytest.mark.parametrize("deterministic", [False, True])
def test_elastic_p2_cell_tiles(n_cells, deterministic):
    """K, f and a second load case of n_cells quadratic cells of two materials (32 cells a block), two clamped
    nodes with prescribed displacements, against the oracle: FP64 sums of a few hundred terms, 1e-12 of the largest."""
    tam = need_gpu()
    pb = meshgen.unit_cube_problem(3, degree=2)
    cells = np.ascontiguousarray(pb.cells[:n_cells])
    used = np.unique(cells)
    back = -np.ones(pb.n_nodes, np.int64)
    back[used] = np.arange(used.size)
    n = used.size
    rng = np.random.default_rng(n_cells)
    mask = np.zeros(n, np.uint8)
    mask[[0, n // 2]] = 1
    q = meshgen.Problem(name="tiles", coords=pb.coords[used], cells=back[cells].astype(np.int32),
                        cell_material=(np.arange(n_cells) % 2).astype(np.int32),
                        mat_props=np.array([[1.0, 0.3, 1e-3], [10.0, 0.2, 2e-3]]), T=rng.random(n), T_ref=0.25,
                        body_force=rng.standard_normal((n, 3)), dirichlet_mask=mask,
                        u_dirichlet=rng.standard_normal((n, 3)))
    d = tam.problem_to_device(q)
    before = tam.set_deterministic_assembly(deterministic)
    try:
        K, rhs = tam.fem_assemble_elasticity(**d)
        load = tam.fem_assemble_load(K, **d)
    finally:
        tam.set_deterministic_assembly(before)
    Ko, fo = fem.assemble_system(q)
    assert sparse_rel(bsr_to_csr(*tam.tam_matrix_export_bsr(K), n_cols_blocks=n), Ko) <= 1e-12
    for f in (rhs, load):
        assert np.abs(f.cpu().numpy().ravel() - fo).max() <= 1e-12 * np.abs(fo).max()
