"""Kernels whose accuracy or edges the calls above them cannot show, called on the library's own symbols: the
float-float grid transform (k_dft.cu) and the factorisation beyond the part of the pivot's row that it
stages at once (k_chol.cu, 512 entries).
"""
import ctypes as ct
import re
import subprocess

import numpy as np
import pytest

import oracle.isdf_oracle as OO

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def symbol(cuda, lib_built):
    names = subprocess.run(["nm", "-D", "--defined-only", str(lib_built)], capture_output=True, text=True, check=True).stdout
    lib = ct.CDLL(str(lib_built))
    return lambda n: getattr(lib, re.search(rf"\b(_ZN4isdf\d+{n}E\w*)", names).group(1))


class CellDev(ct.Structure):
    _fields_ = [("lat", ct.c_double * 9), ("rec", ct.c_double * 9), ("kmesh", ct.c_int * 3), ("mesh", ct.c_int * 3),
                ("lrange", ct.c_int * 3), ("expcut", ct.c_double), ("orthorhombic", ct.c_int)]


def _vp(t):
    return ct.c_void_p(t.data_ptr())


@pytest.mark.parametrize("kmesh,mesh", [
    ((1, 1, 2), (64, 1, 9)), ((1, 5, 7), (11, 13, 17)), ((3, 1, 4), (8, 61, 4)), ((2, 3, 1), (34, 38, 7)),
    ((2, 2, 2), (24, 32, 21)), ((3, 2, 1), (6, 5, 49)), ((2, 2, 2), (64, 64, 3)),
])
def test_float_float_grid_transform(cuda, symbol, kmesh, mesh):
    """Against numpy's FP64 transform.  A float-float operation errs by 2^-44 of its operands, an output of an
    axis of L points is a sum of at most L products in at most two steps, phase and weight add a few more:
    (L_0 + L_1 + L_2 + 24) 2^-44 of the row's 1-norm, times the weight.  FP32 would miss it by 2^20 / sum L."""
    torch = cuda
    lat = np.array([[5.0, 0.1, 0.0], [0.0, 5.3, 0.2], [0.3, 0.0, 4.8]])
    rec = 2 * np.pi * np.linalg.inv(lat).T
    ng, rows, q0, nq = int(np.prod(mesh)), 3, 1, min(2, int(np.prod(kmesh)) - 1)
    rng = np.random.default_rng(1)
    x = rng.standard_normal((nq, rows, ng, 2)) * np.exp(rng.uniform(-4, 4, (nq, rows, 1, 1)))
    hi = x.astype(np.float32)
    lo = (x - hi).astype(np.float32)
    x = hi.astype(np.float64) + lo
    ff = torch.from_numpy(np.ascontiguousarray(np.stack([hi, lo], -1))).cuda()
    c = CellDev()
    c.lat[:], c.rec[:], c.kmesh[:], c.mesh[:] = lat.ravel(), rec.ravel(), kmesh, mesh
    j = np.arange(64)
    ang = np.stack([np.where(j < n, 2 * np.pi * j / n, 0.0) for n in mesh])
    tw = torch.from_numpy(np.cos(ang) - 1j * np.sin(ang)).cuda()
    work = torch.empty(3 * 16 * 64 * 16 + nq * ng * 8, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    assert symbol("grid_coulomb_fft_ff")(ct.c_void_p(0), _vp(ff), ct.c_int(rows), ct.c_int(q0), ct.c_int(nq), ct.byref(c),
                                         _vp(tw), _vp(work)) == 0
    out = ff.cpu().numpy().astype(np.float64).sum(-1)
    out = out[..., 0] + 1j * out[..., 1]
    gi, mk = OO.grid_index_vectors(mesh).astype(np.float64), OO.kmesh_indices(kmesh).astype(np.float64)
    gh = np.where(gi < np.array(mesh) / 2.0, gi, gi - np.array(mesh))
    for i in range(nq):
        m = mk[q0 + i] / np.array(kmesh)
        g = (m[None] + gh) @ rec
        g2 = np.einsum("ij,ij->i", g, g)
        w = np.where(g2 > 1e-300, np.sqrt(4 * np.pi / np.maximum(g2, 1e-300)), 0.0) / ng
        z = (x[i, ..., 0] + 1j * x[i, ..., 1]) * np.exp(-2j * np.pi * (gi / np.array(mesh)) @ m)
        ref = np.fft.fftn(z.reshape((-1,) + mesh), axes=(1, 2, 3)).reshape(rows, ng) * w
        bound = (sum(mesh) + 24) * 2.0 ** -44 * np.abs(z).sum(1)[:, None] * w[None] + 1e-300
        assert (np.abs(out[i] - ref) <= bound).all()


@pytest.mark.parametrize("n,neff,nq", [(513, 513, 1), (600, 530, 3), (700, 700, 2)])
def test_factorisation_beyond_the_staged_row(cuda, symbol, n, neff, nq):
    """Pivots equal the oracle's; L L^H = A to 4 (n + 2) units of the largest diagonal (a complex sum of n products
    and the squares of its terms); the same L on the rows in use when rows that were pivots are left out; and
    W L_S = 1 to 4 (n + 2) units of |W| |L_S|."""
    torch = cuda
    rng = np.random.default_rng(n)
    nk, A = nq + 1, []
    for _ in range(nk):
        b = rng.standard_normal((neff, neff)) + 1j * rng.standard_normal((neff, neff))
        s = 10.0 ** rng.uniform(-2, 0, neff)
        full = np.zeros((n, n), np.complex128)
        full[:neff, :neff] = s[:, None] * (b @ b.conj().T / neff + 0.5 * np.eye(neff)) * s
        A.append(0.5 * (full + full.conj().T))
    qs = list(range(1, nq + 1))
    dA = torch.from_numpy(np.stack(A)).cuda()
    ql = torch.tensor(qs, dtype=torch.int32, device="cuda")
    res = []
    for live in (False, True):
        Lt = torch.zeros_like(dA)
        perm, rank = (torch.zeros(s, dtype=torch.int32, device="cuda") for s in ((nk, n), (nk,)))
        torch.cuda.synchronize()
        assert symbol("pchol_batched")(ct.c_void_p(0), _vp(dA), ct.c_int(n), ct.c_int(neff), ct.c_bool(live), _vp(ql),
                                       ct.c_int(nq), ct.c_double(1e-13), _vp(Lt), _vp(perm), _vp(rank)) == 0
        torch.cuda.synchronize()
        res.append([t.cpu().numpy() for t in (Lt, perm, rank)])
        if live:
            W, work, tmp = (torch.zeros_like(dA) for _ in range(3))
            torch.cuda.synchronize()
            assert symbol("trinv_batched")(ct.c_void_p(0), _vp(Lt), _vp(perm), _vp(rank), ct.c_int(n), ct.c_int(nk),
                                           _vp(ql), ct.c_int(nq), _vp(W), _vp(work), _vp(tmp)) == 0
            torch.cuda.synchronize()
            W = W.cpu().numpy()
    for q in qs:
        (Lt, perm, rank), (Lv, pv, rv) = ([r[i][q] for i in range(3)] for r in res)
        assert rank == neff and rv == neff and np.array_equal(perm, pv)
        assert np.array_equal(perm[:neff], OO.pchol(A[q][:neff, :neff], 1e-13)[1])
        L, tol = Lt[:neff].T, 4 * (n + 2) * U
        assert np.abs(L @ L.conj().T - A[q]).max() <= tol * A[q].real.max()
        p = perm[:neff]
        Ls = np.tril(Lt[:neff][:, p].T)
        assert np.array_equal(Ls, np.tril(Lv[:neff][:, p].T))
        Ws = W[q][:neff][:, p]
        assert (np.abs(Ws @ Ls - np.eye(neff)) <= tol * (np.abs(Ws) @ np.abs(Ls)) + 1e-300).all()
