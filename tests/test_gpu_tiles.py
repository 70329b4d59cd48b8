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


@pytest.mark.parametrize("n", [1, 31, 63, 65, 2 ** 17 + 1])
@pytest.mark.parametrize("width,depth,offset", [(3, 1, 0), (33, 2, 0), (64, 3, 1), (96, 1, 0), (128, 3, 0), (128, 4, 1)])
def test_network_row_and_column_tiles(n, width, depth, offset):
    """FP32 forward pass and gradient at the edges of the 64- and 32-row tiles, of a piece of 2^17 rows, and for
    every column tile (widths 3 to 128, rows that start off a 16-byte boundary when offset is 1), against the FP64
    oracle: sums of at most 128 products in FP32 (forward 1e-5), and over the rows besides (gradient 1e-4)."""
    tam = need_gpu()
    net = tam.Mlp(8, width, depth, 3, seed=5)
    shapes = omlp.layer_shapes(8, width, depth, 3)
    rng = np.random.default_rng(n)
    shift, scale = rng.standard_normal(8).astype(np.float32) * 0.1, (1.0 + rng.random(8)).astype(np.float32)
    out_scale = np.array([0.5, 2.0, 1.5], np.float32)
    net.set_normalization(shift, scale, out_scale)
    theta = net.get_params().astype(np.float64)
    flat = torch.from_numpy(rng.standard_normal(8 * n + offset).astype(np.float32)).cuda()
    X = flat[offset:].view(n, 8)
    Y = torch.from_numpy(rng.standard_normal((n, 3)).astype(np.float32)).cuda()
    args = (shift.astype(np.float64), scale.astype(np.float64), out_scale.astype(np.float64))
    ref, _ = omlp.forward(theta, shapes, X.cpu().numpy().astype(np.float64), *args)
    got = net.forward(X).cpu().numpy()
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max() + 1e-6
    if n < 2 ** 17:
        loss_o, g_o = omlp.loss_and_grad(theta, shapes, X.cpu().numpy().astype(np.float64),
                                         Y.cpu().numpy().astype(np.float64), *args)
        for _ in range(2):  # the second call reuses the workspace
            loss, g = net.loss_grad(X, Y)
            assert abs(loss - loss_o) <= 1e-5 * loss_o
            assert np.linalg.norm(g - g_o) <= 1e-4 * np.linalg.norm(g_o)


@pytest.mark.parametrize("hexes", [(1, 1, 1), (3, 1, 3), (2, 2, 2), (3, 3, 3), (5, 5, 5), (8, 8, 7)])
def test_dense_inverse_tiles(hexes):
    """A K of at most 2,000 unknowns is its own coarsest level, so one V-cycle is K^-1 r: 24 unknowns (less than
    a 32-wide panel), 96 and 192 (whole panels), 81, 648 and 1,944 (a ragged last one).  FP64 elimination of
    matrices with condition numbers below 1e6: 1e-9."""
    tam = need_gpu()
    nx, ny, nz = hexes
    coords, cells = meshgen.box_kuhn(nx, ny, nz)
    n = coords.shape[0]
    q = meshgen.Problem(name="dense", coords=coords, cells=cells, cell_material=np.zeros(len(cells), np.int32),
                        mat_props=np.array([[1.0, 0.3, 1e-3]]), T=None, T_ref=0.0, body_force=None,
                        dirichlet_mask=(coords[:, 0] == 0).astype(np.uint8), u_dirichlet=None)
    d = tam.problem_to_device(q)
    K, _ = tam.fem_assemble_elasticity(**d)
    H = tam.amg_setup(K, d["coords"])
    assert tam.amg_info(H)["n_levels"] == 1
    r = np.random.default_rng(1).standard_normal((n, 3))
    z = tam.amg_vcycle(H, torch.from_numpy(r).cuda()).cpu().numpy().ravel()
    Ko, _ = fem.assemble_system(q)
    ref = np.linalg.solve(Ko.toarray(), r.ravel())
    assert np.linalg.norm(z - ref) <= 1e-9 * np.linalg.norm(ref)


def test_dense_inverse_of_a_nonsymmetric_operator():
    """A heat problem of 125 unknowns (its own coarsest level) whose Jacobian is not symmetric: with the inverse of
    the whole matrix every Newton step's CG ends at once, and the solution is the oracle's."""
    tam = need_gpu()
    pb = meshgen.unit_cube_problem(4)
    faces = meshgen.boundary_faces(pb.cells)
    tp = meshgen.ThermalProblem(pb.coords, pb.cells, pb.cell_material, np.array([[1.0, 1.0, 5e-4, 0.05, 2e-3]]), faces,
                                np.full(len(faces), -1.0), 300.0 + 300.0 * pb.coords[:, 2])
    d = tam.thermal_to_device(tp)
    th = tam.Thermal(d["coords"], d["cells"], d["cell_material"], tp.thermal_props, d["faces"])
    T = torch.full((pb.n_nodes,), 400.0, dtype=torch.float64, device="cuda")
    st = th.newton(T, beta=d["beta"], T_bc=d["T_bc"], rtol=1e-11, lin_rtol=1e-9, reuse=0)
    assert st["linear"] <= 2 * st["newton"]
    To = oth.newton(tp, np.full(pb.n_nodes, 400.0), rtol=1e-11)[0]
    assert np.abs(T.cpu().numpy() - To).max() <= 1e-8 * np.abs(To).max()


@pytest.mark.parametrize("hexes,degree", [((1, 1, 1), 1), ((3, 2, 2), 1), ((4, 3, 3), 2), ((44, 38, 38), 1), ((24, 20, 18), 2)])
def test_vectors_off_a_16_byte_boundary(hexes, degree):
    """x, b and y may start anywhere a float64 may: the same bits as from 16-byte aligned copies, for meshes that
    take the lanes-per-row kernels and ones that take thread-per-row."""
    tam = need_gpu()
    pb = meshgen.slab_box_problem(*hexes, degree=degree)
    d = tam.problem_to_device(pb)
    before = tam.set_deterministic_assembly(True)
    try:
        K, rhs = tam.fem_assemble_elasticity(**d)
        moved = torch.empty(d["cells"].numel() + 1, dtype=torch.int32, device="cuda")[1:].view(d["cells"].shape)
        moved.copy_(d["cells"])
        K2, rhs2 = tam.fem_assemble_elasticity(**dict(d, cells=moved))
    finally:
        tam.set_deterministic_assembly(before)
    assert torch.equal(rhs, rhs2)
    assert torch.equal(tam.tam_matrix_export_bsr(K)[2], tam.tam_matrix_export_bsr(K2)[2])
    n = pb.n_nodes
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn((n, 3), dtype=torch.float64, device="cuda", generator=g)

    def off(v):
        w = torch.empty(v.numel() + 1, dtype=torch.float64, device="cuda")[1:].view(v.shape)
        return w.copy_(v)

    assert torch.equal(tam.tam_matrix_spmv(K, x), tam.tam_matrix_spmv(K, off(x), off(x)))
    assert tam.tam_matrix_residual_norm(K, rhs, x) == tam.tam_matrix_residual_norm(K, off(rhs), off(x))
    H = tam.amg_setup(K, d["coords"])
    assert torch.equal(tam.amg_vcycle(H, x), tam.amg_vcycle(H, off(x), off(x)))
    if tam.amg_info(H)["n_levels"] > 1:
        assert torch.equal(tam.amg_smooth(H, rhs, x.clone(), 3), tam.amg_smooth(H, off(rhs), off(x), 3))


@pytest.mark.parametrize("n_rhs", [(1, 3), (8, 9), (16, 2)])
def test_batch_right_hand_side_tiles(n_rhs):
    """Batched solves with right-hand-side counts at and off the padding to 8 and 16, on a linear and a quadratic
    mesh of several levels, against single solves of each case: both to 1e-10, condition numbers below 1e6, so
    the solutions agree to 1e-5 of their norm (1e-4 of the tolerance times the condition number)."""
    tam = need_gpu()
    rng = np.random.default_rng(3)
    hs, bs, xs = [], [], []
    for (hexes, degree), m in zip((((17, 9, 7), 1), ((9, 5, 4), 2)), n_rhs):
        pb = meshgen.slab_box_problem(*hexes, degree=degree)
        d = tam.problem_to_device(pb)
        K, rhs = tam.fem_assemble_elasticity(**d)
        hs.append(tam.amg_setup(K, d["coords"], tam.amg_params_default(level_precision=1)))
        B = torch.from_numpy(rng.standard_normal((m, 3 * pb.n_nodes))).cuda()
        B.view(m, -1, 3)[:, d["dirichlet_mask"] != 0] = 0.0
        B[-1] = rhs.reshape(-1)
        bs.append(B)
        xs.append(torch.zeros_like(B))
    iters, rels, st = tam.amg_pcg_solve_batch(hs, bs, xs, rtol=1e-10)
    assert st == tam.TAM_OK and max(rels) <= 2e-10
    for H, B, X in zip(hs, bs, xs):
        for b, x in zip(B, X):
            y = torch.zeros_like(b)
            tam.amg_pcg_solve(H, b, y, rtol=1e-10)
            assert float((x - y).norm()) <= 1e-5 * float(y.norm())


@pytest.mark.parametrize("n", [0, 1, 4095, 4096, 4097, 40960, 40961, 70001])
def test_scan_lengths(n):
    """Meshes of n isolated nodes beside one cell: the pattern's scans at one tile, several tiles of one block and
    the three-launch path must give every row one block (the cell's four nodes: 4)."""
    tam = need_gpu()
    coords = np.concatenate([np.array([[0.0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]]), np.full((n, 3), 5.0)])
    q = meshgen.Problem(name="scan", coords=coords, cells=np.array([[0, 1, 2, 3]], np.int32),
                        cell_material=np.zeros(1, np.int32), mat_props=np.array([[1.0, 0.3, 1e-3]]), T=None, T_ref=0.0,
                        body_force=None, dirichlet_mask=np.zeros(n + 4, np.uint8), u_dirichlet=None)
    K, _ = tam.fem_assemble_elasticity(**tam.problem_to_device(q))
    rp = tam.tam_matrix_export_bsr(K)[0].cpu().numpy()
    assert np.array_equal(np.diff(rp), np.r_[np.full(4, 4), np.ones(n, int)])


@pytest.mark.parametrize("precision,tol", [(1, 1e-5), (2, 5e-2)])
@pytest.mark.parametrize("hexes,degree", [((5, 4, 3), 1), ((24, 20, 18), 1), ((36, 30, 30), 1), ((44, 38, 38), 1), ((12, 12, 10), 2)])
def test_low_precision_vcycle_lane_layouts(hexes, degree, precision, tol):
    """One FP32 V-cycle against the FP64 one, for meshes whose levels take 2, 4, 8 and more lanes per row, block
    rows and thread-per-row (FP32 rounding: 1e-5; BF16 finest values: 5e-2)."""
    tam = need_gpu()
    pb = meshgen.slab_box_problem(*hexes, degree=degree)
    d = tam.problem_to_device(pb)
    K, rhs = tam.fem_assemble_elasticity(**d)
    r = torch.randn((pb.n_nodes, 3), dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    z = [tam.amg_vcycle(tam.amg_setup(K, d["coords"], tam.amg_params_default(level_precision=p, coarse_max_dofs=60)), r)
         for p in (0, precision)]
    assert float((z[1] - z[0]).norm() / z[0].norm()) <= tol


@pytest.mark.parametrize("hexes,degree", [((24, 20, 18), 1), ((44, 38, 38), 1), ((20, 20, 20), 2)])
def test_direction_split_beforehand(hexes, degree):
    """The CG's products on rows of several lanes, thread-per-row and two warps per slice: the true residual (plain
    double-float or FP64 product of the result) is what the recurrence says, to a few 2^-48 of its terms."""
    tam = need_gpu()
    pb = meshgen.slab_box_problem(*hexes, degree=degree)
    d = tam.problem_to_device(pb)
    K, rhs = tam.fem_assemble_elasticity(**d)
    H = tam.amg_setup(K, d["coords"])
    x = torch.zeros_like(rhs)
    it, rel, st = tam.amg_pcg_solve(H, rhs, x, rtol=1e-8, max_iter=300)
    true = tam.tam_matrix_residual_norm(K, rhs, x) / float(rhs.norm())
    assert rel <= 1e-8 and abs(true - rel) <= 1e-2 * rel, (it, rel, true)
