"""Interpolation points of orthorhombic cells from the separable Gram (k_basis.cu,
ips_step_kernel) against the oracle's selection, which forms the Gram from Phi.

The indices are integers and must be equal.  Sizes sit at the edges of the
launch: grids below one warp per block, blocks that straddle (g0, g1) rows, an
axis of one point, several terms per AO (contracted shells) with term tiles that
do not divide them, 256-row pieces of the factor, and a selection that runs out
of rank.
"""
import numpy as np
import pytest

import oracle as O
from paper_2601_16379_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cell(kmesh, mesh, contracted=False):
    ex = (0.4, 1.1, 3.0) if contracted else (0.8,)
    cf = (0.5, 0.4, 0.3) if contracted else (1.0,)
    sh = [W.Shell(0, 0, ex, cf), W.Shell(0, 1, (0.9,), (1.0,)), W.Shell(1, 2, ex, cf), W.Shell(1, 0, (2.0,), (0.6,))]
    cell = W.custom_cell(5.0, [[0.01, 0.02, 0.03], [0.37, 0.52, 0.21]], sh, kmesh, mesh)
    cell.lattice = np.diag([5.0, 5.3, 4.8])
    return cell


@pytest.mark.parametrize("kmesh,mesh,n_p,contracted", [
    ((1, 1, 1), (3, 2, 5), 9, False),
    ((2, 2, 2), (7, 9, 5), 60, True),
    ((3, 1, 2), (1, 31, 33), 50, False),
    ((2, 1, 3), (16, 12, 1), 40, True),
    ((2, 2, 3), (12, 11, 13), 300, False),
    ((1, 2, 1), (40, 33, 35), 20, True),
])
def test_points_equal_the_oracle(cuda, lib_built, kmesh, mesh, n_p, contracted):
    from paper_2601_16379_gb300 import binding as B
    cell = _cell(kmesh, mesh, contracted)
    ref, found = O.select_ips(O.bloch_ao(cell), n_p, 11)
    g = B.Isdf(cell, B.ISDF_FP64)
    if found < n_p:
        with pytest.raises(B.IsdfError) as e:
            g.build_points(n_p, 11)
        assert e.value.code == -4
        n_p = found - 2
    assert np.array_equal(g.build_points(n_p, 11), ref[:n_p])
    g.close()
