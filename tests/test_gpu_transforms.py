"""The small transforms of the fit and metric (k_dft.cu) and the factorisation between them
(k_chol.cu), through V^q, against the oracle.

Axes sit at the edges of the mixed-radix forms: lengths 1 and 2, products of two factors of at most
8, the largest (64), a factor above 8 (11, 13, 17, 34 = 2 x 17, 49 = 7 x 7, 61), grids that are not
a multiple of a block's lines or columns, and k-meshes of every kind of axis, 96 points among them.
FP64_TC takes the direct sums in their place.

Tolerance: X, Pi and eta agree to 1e-13 with the oracle; the solve with tau = 1e-3 multiplies that by
at most 1 / tau, twice in V.  1e-8 of the largest entry of V leaves an order of magnitude.
"""
import numpy as np
import pytest

import oracle as O
from paper_2601_16379_gb300 import workloads as W

pytestmark = pytest.mark.gpu

def _cell(kmesh, mesh):
    sh = [W.Shell(0, 0, (0.6,), (1.0,)), W.Shell(0, 1, (0.9,), (1.0,)), W.Shell(1, 1, (1.4,), (1.0,)),
          W.Shell(1, 2, (1.1,), (0.7,))]
    return W.custom_cell(5.0, [[0.013, 0.022, 0.031], [0.37, 0.52, 0.21]], sh, kmesh, mesh)


def _check(torch, cell, n_p, prec, tau=1e-3, tol=1e-8):
    from paper_2601_16379_gb300 import binding as B
    pts = W.seeded_points(cell, n_p, 3)
    phi = O.bloch_ao(cell)
    X = O.interp_vectors(phi, pts)
    zeta, ranks = O.fit_zeta(O.metric_pi(X, cell.kmesh), O.rhs_eta(X, phi, cell.kmesh), tau)
    ref = O.coulomb_metric(cell, zeta, range(cell.nkpts))
    g = B.Isdf(cell, prec)
    g.set_time_reversal(False)  # q + G in a box is not symmetric: the oracle takes every q as it is
    g.set_points(pts)
    assert np.array_equal(g.fit_zeta(tau), ranks)
    V = torch.empty((cell.nkpts, n_p, n_p), dtype=torch.complex128, device="cuda")
    g.coulomb_metric(V)
    assert np.abs(V.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
    g.close()


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("kmesh,mesh", [
    ((1, 1, 1), (2, 3, 5)),
    ((1, 1, 2), (64, 1, 9)),
    ((1, 5, 7), (11, 13, 17)),
    ((5, 5, 5), (25, 3, 22)),
    ((3, 1, 16), (8, 61, 4)),
    ((9, 11, 1), (6, 5, 49)),
    ((2, 13, 1), (34, 38, 7)),
    ((15, 1, 14), (7, 8, 16)),
    ((4, 4, 6), (9, 8, 10)),
    ((12, 2, 1), (37, 4, 33)),
])
def test_metric_on_edge_meshes(cuda, lib_built, kmesh, mesh, prec):
    _check(cuda, _cell(kmesh, mesh), min(14, int(np.prod(mesh)) // 3), prec)


@pytest.mark.parametrize("n_p", [1, 2, 15, 16, 17, 31, 33, 63, 64, 65, 127, 129, 200])
def test_factorisation_sizes(cuda, lib_built, n_p):
    """tau = 1e-6 keeps more pivots than one pass of the factorisation holds; the bound scales with it."""
    _check(cuda, _cell((2, 1, 3), (12, 10, 14)), n_p, 0, tau=1e-6, tol=1e-5)


@pytest.mark.parametrize("kmesh,mesh", [
    ((1, 1, 2), (64, 1, 9)),
    ((1, 5, 7), (11, 13, 17)),
    ((3, 1, 4), (8, 61, 4)),
    ((2, 3, 1), (34, 38, 7)),
    ((2, 2, 2), (24, 32, 21)),
    ((3, 2, 1), (6, 5, 49)),
])
def test_metric_in_float_float(cuda, lib_built, kmesh, mesh):
    """The mixed path's grid transform: V_xi is cut to four slices (2^-28 of its rows' largest entries),
    which the solve multiplies by up to 1 / tau in sums of at most 14 x 14 terms: 7e-4 of the largest entry."""
    _check(cuda, _cell(kmesh, mesh), min(14, int(np.prod(mesh)) // 3), 1, tol=1e-3)


@pytest.mark.parametrize("n_p", [1, 16, 17, 63, 65, 79, 81, 130])
def test_partial_tiles_of_the_fixed_chains(cuda, lib_built, n_p):
    """xi, V_xi and L of FP64_TC on 64 x 64 tiles of which only some 16-row and 16-column parts are formed."""
    _check(cuda, _cell((2, 1, 3), (12, 10, 14)), n_p, 2, tau=1e-6, tol=1e-5)
