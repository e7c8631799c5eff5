"""Fragment ERIs of the tensor-core paths at the edges of their kernels (k_tc.cu, k_dft.cu) against
the FP64 path of the same handle settings.

Sizes: interpolation points around the 32 and 64 columns of a pass and the 128 rows of a block,
one orbital, fragments whose pair rows straddle a block, a rank below n_p (columns of L without a
pivot), and k-meshes with and without a kernel of their own (96 points among them).  The bounds are
those of the paths: 1e-6 Ha (mixed), 1e-8 Ha (FP64_TC).
"""
import numpy as np
import pytest

from paper_2601_16379_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TAU = 1e-3


def _cell(kmesh):
    sh = [W.Shell(0, 0, (0.6,), (1.0,)), W.Shell(0, 1, (0.9,), (1.0,)), W.Shell(1, 1, (1.4,), (1.0,)),
          W.Shell(1, 2, (1.1,), (0.7,))]
    return W.custom_cell(5.0, [[0.013, 0.022, 0.031], [0.37, 0.52, 0.21]], sh, kmesh, (12, 10, 14))


def _run(torch, cell, prec, n_p, frags, gammas):
    from paper_2601_16379_gb300 import binding as B
    g = B.Isdf(cell, prec)
    g.set_points(W.seeded_points(cell, n_p, 3))
    g.fit_zeta(TAU)
    g.coulomb_metric()
    outs = [torch.empty((f.norb,) * 4, dtype=torch.complex64 if prec == 1 else torch.complex128, device="cuda")
            for f in frags]
    ej, ek = g.fragment_eri([torch.from_numpy(f.C).cuda() for f in frags],
                            [torch.from_numpy(x).cuda() for x in gammas], outs)
    torch.cuda.synchronize()
    g.close()
    return [o.cpu().numpy() for o in outs], np.asarray(ej), np.asarray(ek)


@pytest.mark.parametrize("prec,tol", [(1, 1e-6), (2, 1e-8)])
@pytest.mark.parametrize("kmesh,n_p,norbs", [
    ((2, 1, 3), 5, (1,)),
    ((2, 1, 3), 31, (3, 2)),
    ((2, 2, 2), 33, (11, 1)),
    ((2, 1, 3), 64, (12,)),
    ((3, 3, 3), 65, (5, 5, 5)),
    ((1, 1, 5), 129, (16,)),
    ((2, 1, 1), 200, (17, 4)),
    ((4, 4, 6), 40, (4,)),
])
def test_eri_against_fp64(cuda, lib_built, kmesh, n_p, norbs, prec, tol):
    cell = _cell(kmesh)
    frags = [W.make_fragment(cell, 7, i, n) for i, n in enumerate(norbs)]
    gam = [f.gamma for f in frags]
    ref, rj, rk = _run(cuda, cell, 0, n_p, frags, gam)
    out, ej, ek = _run(cuda, cell, prec, n_p, frags, gam)
    for a, b in zip(out, ref):
        assert np.abs(a - b).max() <= tol
    assert np.abs(ej - rj).max() <= tol and np.abs(ek - rk).max() <= tol


@pytest.mark.parametrize("prec", [1, 2])
def test_traces_of_a_gamma_just_off_hermitian(cuda, lib_built, prec):
    """A gamma that is Hermitian to rounding counts each pair of mirrored blocks twice, any other
    sums both.  An antisymmetric part of 1e-11 takes the second form and moves the traces by no
    more than 1e-9 (a few thousand terms of |gamma| <= 2 and |(pq|rs)| of order 1)."""
    cell = _cell((2, 1, 3))
    frags = [W.make_fragment(cell, 7, 0, 9)]
    gam = frags[0].gamma
    off = gam + 1e-11 * np.triu(np.ones_like(gam), 1)
    _, ej, ek = _run(cuda, cell, prec, 48, frags, [gam])
    _, oj, ok = _run(cuda, cell, prec, 48, frags, [off])
    assert np.abs(ej - oj).max() <= 1e-9 and np.abs(ek - ok).max() <= 1e-9
