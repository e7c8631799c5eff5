"""Point selection of orthorhombic cells that runs out of rank on grids of several waves of blocks
(k_basis.cu, ips_step_kernel): every block of a step has to take the same decision to stop.

The count of points found and the points themselves are integers and equal the oracle's.
"""
import re

import numpy as np
import pytest

import oracle as O
from paper_2601_16379_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cell(kmesh, mesh):
    sh = [W.Shell(0, 0, (0.9,), (1.0,)), W.Shell(1, 1, (1.3,), (1.0,))]
    cell = W.custom_cell(5.0, [[0.01, 0.02, 0.03], [0.37, 0.52, 0.21]], sh, kmesh, mesh)
    cell.lattice = np.diag([5.0, 5.3, 4.8])
    return cell


@pytest.mark.parametrize("kmesh,mesh,chol_tol", [
    ((1, 1, 1), (48, 48, 40), 1e-3),   # 360 blocks
    ((2, 1, 1), (35, 34, 36), 1e-4),   # 168 blocks
    ((1, 1, 2), (9, 10, 11), 1e-3),    # less than a block per SM
])
def test_selection_out_of_rank(cuda, lib_built, kmesh, mesh, chol_tol):
    from paper_2601_16379_gb300 import binding as B
    cell = _cell(kmesh, mesh)
    n_p = 60
    ref, found = O.select_ips(O.bloch_ao(cell), n_p, 5, chol_tol=chol_tol)
    assert 2 < found < n_p
    g = B.Isdf(cell, B.ISDF_FP64)
    for _ in range(20):
        with pytest.raises(B.IsdfError) as e:
            g.build_points(n_p, 5, chol_tol)
        assert e.value.code == -4 and int(re.search(r"after (\d+) of", str(e.value)).group(1)) == found
    assert np.array_equal(g.build_points(found, 5, chol_tol), ref)
    g.close()


def test_more_points_than_a_piece_of_the_factor(cuda, lib_built):
    """600 points: the pivot's row of the factor is staged in pieces of 512.  The residuals keep 5e-13 of the
    largest diagonal away from every tie window (rounding: ~1e-15), so that the indices are determined."""
    from paper_2601_16379_gb300 import binding as B
    sh = [W.Shell(a, l, (x,), (1.0,)) for a in (0, 1) for l, x in ((0, 0.6), (1, 0.9), (2, 1.4))]
    cell = W.custom_cell(5.0, [[0.01, 0.02, 0.03], [0.37, 0.52, 0.21]], sh, (2, 2, 3), (16, 15, 17))
    cell.lattice = np.diag([5.0, 5.3, 4.8])
    ref, found = O.select_ips(O.bloch_ao(cell), 600, 11)
    assert found == 600
    g = B.Isdf(cell, B.ISDF_FP64)
    assert np.array_equal(g.build_points(600, 11), ref)
    g.close()


def test_long_contractions_at_gamma(cuda, lib_built):
    """2000 terms at one k-point go by the pass over Phi: the same points as the oracle's."""
    from paper_2601_16379_gb300 import binding as B
    ex, cf = tuple(np.geomspace(0.4, 30.0, 10)), tuple(np.linspace(0.6, 0.1, 10))
    sh = [W.Shell(a, l, ex, cf) for a in (0, 1) for l in (0, 1, 2)]
    cell = W.custom_cell(5.0, [[0.01, 0.02, 0.03], [0.37, 0.52, 0.21]], sh, (1, 1, 1), (14, 13, 15))
    cell.lattice = np.diag([5.0, 5.3, 4.8])
    ref, found = O.select_ips(O.bloch_ao(cell), 40, 3)
    assert found == 40
    g = B.Isdf(cell, B.ISDF_FP64)
    assert np.array_equal(g.build_points(40, 3), ref)
    g.close()
