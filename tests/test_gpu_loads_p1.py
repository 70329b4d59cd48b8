"""Loads of linear cells with prescribed displacements, cell by cell of a warp.

The load-only kernel skips the stiffness of warps without Dirichlet nodes and,
in the others, the pairs of nodes that no cell of the warp needs.
"""
import numpy as np
import pytest

from gpu_util import bsr_to_csr, need_gpu, sparse_rel
from oracle import fem
from paper_1804_10060_gb300 import meshgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_cells", [1, 31, 32, 33, 127, 128, 129, 300])
@pytest.mark.parametrize("held", ["first", "last", "some", "none"])
@pytest.mark.parametrize("deterministic", [False, True])
def test_elastic_p1_cell_tiles(n_cells, held, deterministic):
    """K, f and a second load case of n_cells linear cells of two materials (32 cells a warp, 128 a block), with
    prescribed displacements on nodes of the first cell, of the last, of every 40th, or none: FP64 sums of a few
    hundred terms against the oracle, 1e-12 of the largest."""
    tam = need_gpu()
    coords, cells = meshgen.box_kuhn(5, 5, 4)
    cells = np.ascontiguousarray(cells[:n_cells])
    used = np.unique(cells)
    back = -np.ones(len(coords), np.int64)
    back[used] = np.arange(used.size)
    cells = back[cells].astype(np.int32)
    n = used.size
    rng = np.random.default_rng(n_cells)
    mask = np.zeros(n, np.uint8)
    mask[{"first": cells[0, :2], "last": cells[-1, 2:3], "some": cells[::40, 1], "none": []}[held]] = 1
    q = meshgen.Problem(name="tiles", coords=coords[used], cells=cells, cell_material=(np.arange(n_cells) % 2).astype(np.int32),
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
