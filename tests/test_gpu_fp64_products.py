"""Plain FP64 products: matrices outside the double-float range, and hierarchies that ask for FP64."""
import numpy as np
import pytest

from gpu_util import bsr_to_csr, exact_spmv, need_gpu, torch
from paper_1804_10060_gb300 import meshgen

pytestmark = pytest.mark.gpu


def _off(v):
    """A copy of v that starts 8 bytes past a 16-byte boundary."""
    w = torch.empty(v.numel() + 1, dtype=torch.float64, device="cuda")[1:].view(v.shape)
    return w.copy_(v)


@pytest.mark.parametrize("hexes,degree", [((1, 1, 1), 1), ((12, 5, 5), 1), ((1, 1, 1), 2), ((9, 4, 3), 2)])
def test_spmv_outside_the_double_float_range(hexes, degree):
    """K of stiffness 2^120: y = K x against exactly summed products.  A row of n products is a chain of n FP64
    multiply-adds: n 2^-53 sum_j |K_ij x_j|; the same bits from vectors off a 16-byte boundary."""
    tam = need_gpu()
    pb = meshgen.slab_box_problem(*hexes, degree=degree)
    d = tam.problem_to_device(pb)
    d["mat_props"][:, 0] *= 2.0 ** 120
    K, _ = tam.fem_assemble_elasticity(**d)
    x = torch.randn((pb.n_nodes, 3), dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    y = tam.tam_matrix_spmv(K, x)
    assert torch.equal(y, tam.tam_matrix_spmv(K, _off(x), _off(x)))
    A = bsr_to_csr(*tam.tam_matrix_export_bsr(K), n_cols_blocks=pb.n_nodes)
    ref, s = exact_spmv(A, x.cpu().numpy().ravel())
    n = np.diff(A.indptr).max() + 3
    assert (np.abs(y.cpu().numpy().ravel() - ref) <= n * 2.0 ** -53 * s).all()


@pytest.mark.parametrize("hexes,degree", [((9, 4, 3), 2), ((24, 20, 18), 1), ((24, 20, 18), 2), ((44, 38, 38), 1)])
def test_fp64_vcycle_off_a_16_byte_boundary(hexes, degree):
    """spmv_fp64 = 1: the same bits for any alignment, on block-CSR rows, the lanes-per-row store and SELL."""
    tam = need_gpu()
    pb = meshgen.slab_box_problem(*hexes, degree=degree)
    d = tam.problem_to_device(pb)
    K, rhs = tam.fem_assemble_elasticity(**d)
    H = tam.amg_setup(K, d["coords"], tam.amg_params_default(spmv_fp64=1))
    x = torch.randn((pb.n_nodes, 3), dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    assert torch.equal(tam.amg_vcycle(H, x), tam.amg_vcycle(H, _off(x), _off(x)))
    assert torch.equal(tam.amg_smooth(H, rhs, x.clone(), 3), tam.amg_smooth(H, _off(rhs), _off(x), 3))
