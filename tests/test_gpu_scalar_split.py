"""Heat problems whose level 0 runs thread per row (65,536 rows and more): the products read vectors split
beforehand, a second copy of every iterate that has to stay in step with it through the smoother's swaps, the
prolongation and the CG's directions."""
import numpy as np
import pytest

from gpu_util import need_gpu, torch
from paper_1804_10060_gb300 import meshgen

pytestmark = pytest.mark.gpu


def _step_pair(tam, pb, tp, **prm):
    """A steady solve, then a backward-Euler step on the same (kept) hierarchy: temperatures and statistics."""
    d = tam.thermal_to_device(tp)
    th = tam.Thermal(d["coords"], d["cells"], d["cell_material"], tp.thermal_props, d["faces"], d["dirichlet_mask"],
                     tam.amg_params_default(**prm))
    T = torch.full((pb.n_nodes,), 400.0, dtype=torch.float64, device="cuda")
    out = []
    for kw in (dict(), dict(T_old=None, dt=0.01, theta=1.0)):
        if kw:
            kw["T_old"] = out[0][0]
            T = T + 20.0 * d["coords"][:, 0]
        st = th.newton(T, beta=d["beta"], T_bc=d["T_bc"], T_dirichlet=d["T_dirichlet"], rtol=1e-11, lin_rtol=1e-10,
                       reuse=1, **kw)
        assert st["status"] == 0 and st["rel"] <= 1e-11, st
        out.append((T.clone(), st["linear"]))
    th.destroy()
    return out


# 41^3 nodes: two warps a slice; 93^3: one.  The held layers give slices of one-entry rows beside full ones.
@pytest.mark.parametrize("n,degree,held,prm", [
    (40, 1, 0.2, {}), (40, 1, 0.2, dict(smoother_degree=1, small_level_degree=1)), (40, 1, 0.0, dict(smoother_degree=3)),
    (40, 1, 0.0, dict(spmv_fp64=2)), (20, 2, 0.2, {}), (20, 2, 0.0, dict(smoother_degree=3)), (92, 1, 0.1, {})])
def test_split_vectors(n, degree, held, prm):
    """Against the same Newton solves in plain FP64 (spmv_fp64 = 1), which split nothing: both to ||F|| <= 1e-11
    ||F_0||, so the temperatures agree to 1e-8, and as many CG iterations to a tenth (double-float products keep
    2^-45 of a row's sum; FP32 rounding of an iterate that fell out of step would cost the convergence)."""
    tam = need_gpu()
    pb = meshgen.unit_cube_problem(n, degree=degree)
    assert pb.n_nodes >= 65536
    faces = meshgen.boundary_faces(pb.cells)
    z = pb.coords[:, 2]
    tp = meshgen.ThermalProblem(pb.coords, pb.cells, pb.cell_material, np.array([[1.0, 1.0, 5e-4, 0.05, 5e-5]]), faces,
                                np.full(len(faces), -1.0), 300.0 + 300.0 * z)
    if held:
        tp.dirichlet_mask = (z <= held).astype(np.uint8)
        tp.T_dirichlet = np.full(pb.n_nodes, 350.0)
    got = _step_pair(tam, pb, tp, **prm)
    ref = _step_pair(tam, pb, tp, **dict(prm, spmv_fp64=1))
    for (T, it), (R, ir) in zip(got, ref):
        assert float((T - R).abs().max()) <= 1e-8 * float(R.abs().max())
        assert abs(it - ir) <= max(2, ir // 10), (it, ir)
