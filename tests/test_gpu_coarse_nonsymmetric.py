"""Hierarchies of a heat Jacobian that is not symmetric (kappa depends on T).

Every R J P of such a hierarchy is non-symmetric too, and the coarsest one must
be inverted as it is.  One linear solve of a Newton step is compared with the
same CG on the CPU: the oracle's hierarchy of the same Jacobian (the GPU's:
aggregation is unique) with the inverse of the whole coarsest operator.
"""
import numpy as np
import pytest

from gpu_util import need_gpu, torch
from oracle import amg as oamg
from oracle import thermal as oth
from paper_1804_10060_gb300 import meshgen

pytestmark = pytest.mark.gpu

TAM_ERR_NOT_CONVERGED = -5
PARAMS = dict(strength_theta=0.0, coarse_max_dofs=500, coarse_min_dofs=0)


def _oracle_hierarchy(J, monkeypatch):
    def inverse(A):
        A = A.toarray()
        assert len(A) > 32  # more than one tile of the GPU's elimination
        # pivots of the elimination without pivoting: positive, the GPU accepts the operator
        U, pivots = A.copy(), []
        for k in range(len(U)):
            pivots.append(U[k, k])
            U[k + 1:, k + 1:] -= np.outer(U[k + 1:, k] / U[k, k], U[k, k + 1:])
        assert min(pivots) > 1e-2 * max(pivots)
        return np.linalg.inv(A)

    monkeypatch.setattr(oamg, "coarse_inverse", inverse)
    return oamg.setup(J, np.ones((J.shape[0], 1)), 1, theta=0.0, coarse_max_dofs=500, coarse_min_dofs=0)


@pytest.mark.parametrize("n,hi,axis,reverse", [(8, 300.0, 2, False), (12, 300.0, 0, True), (12, 300.0, 2, False),
                                               (16, 100.0, 2, True), (16, 200.0, 0, False)])
def test_cg_of_a_strongly_nonsymmetric_jacobian(n, hi, axis, reverse, monkeypatch):
    """kappa = 0.05 + 2e-3 T under a steep T: coarsest levels of 38, 107 and 216 unknowns.  As many CG iterations as
    the oracle's, with a fifth (at least 2) allowed for rounding, which CG on a non-symmetric matrix amplifies (with the tiles below the diagonal mirrored: 45 iterations
    for 18, 22 for 19, 16 for 13)."""
    tam = need_gpu()
    pb = meshgen.unit_cube_problem(n)
    faces = meshgen.boundary_faces(pb.cells)
    x = pb.coords[:, axis]
    T0 = hi * (1.0 - x if reverse else x)
    T_bc = T0 + 100.0 * np.random.default_rng(n).standard_normal(pb.n_nodes)
    tp = meshgen.ThermalProblem(pb.coords, pb.cells, pb.cell_material, np.array([[1.0, 1.0, 5e-4, 0.05, 2e-3]]), faces,
                                np.full(len(faces), -1.0), T_bc)
    F, J = oth.assemble_thermal(tp, T0)
    Ho = _oracle_hierarchy(J, monkeypatch)
    assert len(Ho.levels) > 1
    A = Ho.levels[-1].A
    assert abs(A - A.T).max() > 1e-2 * abs(A).max()
    _, it_o, rel_o = oamg.pcg(J, F, Ho, rtol=1e-8, max_iter=100)
    assert rel_o <= 2e-8
    d = tam.thermal_to_device(tp)
    th = tam.Thermal(d["coords"], d["cells"], d["cell_material"], tp.thermal_props, d["faces"],
                     params=tam.amg_params_default(**PARAMS))
    T = torch.from_numpy(T0).cuda()
    st = th.newton(T, beta=d["beta"], T_bc=d["T_bc"], rtol=1e-14, max_newton=1, lin_rtol=1e-8, lin_max_iter=100, reuse=0,
                   raise_on_error=False)
    assert st["status"] == TAM_ERR_NOT_CONVERGED and st["newton"] == 1, st  # the one step asked for was taken
    assert 0 < st["linear"] <= it_o + max(2, it_o // 5), (st, it_o)
