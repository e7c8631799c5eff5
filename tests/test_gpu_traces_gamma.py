"""E_J and E_K of the tensor-core paths (k_tc.cu, syrk_eri_kernel) around the size from which gamma is tested for
being Hermitian, against the traces formed from the returned integrals.

A Hermitian gamma gives the documented traces.  Another gamma is taken as the sum over the ordered blocks of pairs
reads it (gamma_pq of the row pair with p <= q, gamma_yx of the column pair); counting mirrored blocks twice would
then give a different number, by a large part of it.

Tolerance: FP64 sums over complex128 integrals (FP64_TC) of at most n^4 terms that cancel, 1e-12 of the sum of
their magnitudes; complex64 integrals (mixed) add 2^-24 of it.
"""
import numpy as np
import pytest

from paper_2601_16379_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cell():
    sh = [W.Shell(0, 0, (0.6,), (1.0,)), W.Shell(0, 1, (0.9,), (1.0,)), W.Shell(1, 1, (1.4,), (1.0,)),
          W.Shell(1, 2, (1.1,), (0.7,))]
    return W.custom_cell(5.0, [[0.013, 0.022, 0.031], [0.37, 0.52, 0.21]], sh, (2, 2, 3), (8, 7, 9))


def _block_traces(eri, g):
    """(E_J, E_K, sum of magnitudes) over the ordered pairs of orbits (p <= q), (x <= y), as the kernel reads gamma."""
    n = len(g)
    p, q = np.triu_indices(n)
    ej = ek = mag = 0.0
    for x, y in zip(*np.triu_indices(n)):
        r1, r2 = eri[p, q, y, x], eri[p, q, x, y]
        A, B = g[p, q], g[y, x]
        pr, pc = p != q, x != y
        # the four orders of a block: A r, conj(A) and so on reduce to 4 Re, 2 Re or 1 by what is diagonal
        if pc:
            aj = np.where(pr, 2 * ((A * B * r1).real + (A * np.conj(B) * r2).real), 2 * (g[p, p].real * (B * r1).real))
            ak = np.where(pr, 2 * ((g[p, x] * g[y, q] * r1).real + (g[p, y] * g[x, q] * r2).real),
                          2 * (g[p, x] * g[y, p] * r1).real)
        else:
            aj = np.where(pr, 2 * g[x, x].real * (A * r1).real, g[p, p].real * g[x, x].real * r1.real)
            ak = np.where(pr, 2 * (g[p, x] * g[x, q] * r1).real, np.abs(g[p, x]) ** 2 * r1.real)
        ej += aj.sum()
        ek += ak.sum()
        mag += np.abs(aj).sum() + np.abs(ak).sum()
    return 0.5 * ej, -0.25 * ek, mag


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("n", [9, 47, 48, 61])
def test_traces_of_any_gamma(cuda, lib_built, n, prec):
    from paper_2601_16379_gb300 import binding as B
    torch = cuda
    cell = _cell()
    f = W.make_fragment(cell, 7, 0, n)
    rng = np.random.default_rng(n)
    skew = f.gamma + 0.5 * (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    g = B.Isdf(cell, prec)
    g.set_points(W.seeded_points(cell, 60, 3))
    g.fit_zeta(1e-5)
    g.coulomb_metric()
    eri = torch.empty((n,) * 4, dtype=torch.complex64 if prec == 1 else torch.complex128, device="cuda")
    tol = 2.0 ** -24 if prec == 1 else 1e-12
    for gam, hermitian in ((f.gamma, True), (skew, False)):
        ej, ek = g.fragment_eri([torch.from_numpy(f.C).cuda()], [torch.from_numpy(gam).cuda()], [eri])
        e = eri.cpu().numpy().astype(np.complex128)
        rj, rk, mag = _block_traces(e, gam)
        assert abs(ej[0] - rj) <= tol * mag and abs(ek[0] - rk) <= tol * mag
        if hermitian:
            dj = 0.5 * np.einsum("pq,rs,pqrs->", gam, gam, e, optimize=True).real
            dk = -0.25 * np.einsum("ps,rq,pqrs->", gam, gam, e, optimize=True).real
            assert abs(ej[0] - dj) <= tol * mag and abs(ek[0] - dk) <= tol * mag
        else:
            # each unordered pair of orbits once, off-diagonal ones twice: what the doubled form would return
            lower = _doubled(e, gam)
            assert abs(lower - rj) > 1e3 * tol * mag
    g.close()


def _doubled(eri, g):
    """E_J with the block of the later row orbit counted twice instead of its mirror."""
    n = len(g)
    p, q = np.triu_indices(n)
    ej = 0.0
    for o2, (x, y) in enumerate(zip(p, q)):
        s = slice(o2, None)
        r1, r2 = eri[p[s], q[s], y, x], eri[p[s], q[s], x, y]
        A, B, pr = g[p[s], q[s]], g[y, x], p[s] != q[s]
        if x != y:
            aj = np.where(pr, 2 * ((A * B * r1).real + (A * np.conj(B) * r2).real), 2 * (g[p[s], p[s]].real * (B * r1).real))
        else:
            aj = np.where(pr, 2 * g[x, x].real * (A * r1).real, g[p[s], p[s]].real * g[x, x].real * r1.real)
        ej += 2 * aj.sum() - aj[0]
    return 0.5 * ej
