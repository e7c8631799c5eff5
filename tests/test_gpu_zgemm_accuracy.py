"""Accuracy of the complex128 tensor-core product (k_ztc.cu) against the FP64 FMA chain (k_gemm.cu), both called
directly, with sums in extended precision as the reference.

The operands are those that tell the two apart: Gaussian, with columns that decay along k (Fourier
coefficients), with rows of very different size, and with opposite grading of k in the two operands (the
inverse factor and the factor of L = W^T L_xi), which the caller undoes by powers of two.

Bounds.  (1) Per component |C - exact| <= K 2^-55.9 max|a_i| max|b_j| + 2^-53 |C|: digits are scaled to
[32, 64), so that the dropped digit products are at most 7.03 x 2^14 x 2^-64 and the two roundings 2^-50
each way, 8.03 x 2^-60 of max|a_i| max|b_j| >= 2^10 in all, twice per component.  (2) The root mean square
error is no larger than the chain's.
"""
import ctypes as ct
import re
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LD = np.longdouble


class ZOpt(ct.Structure):
    _fields_ = [("lowerA", ct.c_int), ("brow", ct.c_void_p), ("sIdx", ct.c_int64), ("qmap", ct.c_void_p),
                ("krank", ct.c_void_p), ("slices", ct.c_int), ("kexp", ct.c_void_p), ("sExp", ct.c_int64),
                ("kneg", ct.c_int)]


@pytest.fixture(scope="module")
def products(cuda, lib_built):
    """(product(op A, op B, A, B, kexp, kneg, tensor cores)) on the library's own symbols."""
    torch = cuda
    names = subprocess.run(["nm", "-D", "--defined-only", str(lib_built)], capture_output=True, text=True, check=True).stdout
    lib = ct.CDLL(str(lib_built))
    fn = lambda n: getattr(lib, re.search(rf"\b(_ZN4isdf\d+{n}E\w*)", names).group(1))  # noqa: E731
    ztc, zg, wb = fn("zgemm_tc"), fn("zgemm"), fn("zgemm_tc_work_bytes")
    wb.restype = ct.c_size_t
    i64, vp = ct.c_int64, ct.c_void_p
    err = torch.zeros(4, dtype=torch.int32, device="cuda")

    def run(opA, opB, A, B, kexp=None, kneg=0, tc=True):
        a, b = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A, B))
        m, k = A.shape if opA in "NR" else A.shape[::-1]
        n = B.shape[1] if opB in "NR" else B.shape[0]
        c = torch.zeros(m, n, dtype=torch.complex128, device="cuda")
        o = ZOpt(slices=8)
        if kexp is not None:
            kx = torch.from_numpy(np.ascontiguousarray(kexp, np.int32)).cuda()
            o.kexp, o.sExp, o.kneg = kx.data_ptr(), k, kneg
        args = [vp(0), ct.c_char(opA.encode()), ct.c_char(opB.encode()), ct.c_int(m), ct.c_int(n), ct.c_int(k),
                ct.c_double(1.0), vp(a.data_ptr()), i64(A.shape[1]), i64(0), vp(b.data_ptr()), i64(B.shape[1]), i64(0),
                vp(c.data_ptr()), i64(n), i64(0), ct.c_int(1), ct.byref(o)]
        torch.cuda.synchronize()
        if tc:
            size = wb(8, m, n, k, 1, False)
            work = torch.empty(size, dtype=torch.uint8, device="cuda")
            assert ztc(*args, vp(work.data_ptr()), ct.c_size_t(size), vp(err.data_ptr())) == 0
        else:
            assert zg(*args) == 0
        torch.cuda.synchronize()
        assert int(err[0]) == 0
        return c.cpu().numpy()

    return run


def _op(x, op):
    x = x.T if op in "TC" else x
    return x.conj() if op in "CR" else x


def _exact(A, B):
    ar, ai, br, bi = (np.ascontiguousarray(v).astype(LD) for v in (A.real, A.imag, B.real, B.imag))
    re_, im = np.zeros((2, A.shape[0], B.shape[1]), LD)
    for k in range(A.shape[1]):
        re_ += np.outer(ar[:, k], br[k]) - np.outer(ai[:, k], bi[k])
        im += np.outer(ar[:, k], bi[k]) + np.outer(ai[:, k], br[k])
    return re_, im


def _err(C, ex):
    return np.maximum(np.abs(C.real.astype(LD) - ex[0]), np.abs(C.imag.astype(LD) - ex[1])).astype(np.float64)


def _amax(x, axis):
    return np.maximum(np.abs(x.real), np.abs(x.imag)).max(axis)


def _operands(kind, m, n, k, seed):
    rng = np.random.default_rng(seed)
    g = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    A, B, d = g(m, k), g(k, n), None
    if kind == "decay":
        f = 1.0 / (1.0 + np.arange(k)) ** 1.5
        A, B = A * f, B * f[:, None]
    elif kind == "rows":
        A, B = A * 2.0 ** rng.uniform(-30, 30, (m, 1)), B * 2.0 ** rng.uniform(-30, 30, (1, n))
    elif kind == "graded":
        d = np.floor(24 * np.arange(k) / k).astype(int)
        A, B = A * 2.0 ** d, B * 2.0 ** -d[:, None].astype(float)
    return A, B, d


@pytest.mark.parametrize("kind", ["plain", "decay", "rows", "graded"])
@pytest.mark.parametrize("m,n,k,ops", [
    (5, 7, 6, "NN"), (64, 32, 26, "RT"), (33, 65, 32, "NC"), (64, 33, 33, "TN"), (40, 40, 52, "CN"),
    (70, 31, 119, "TN"), (32, 64, 143, "NN"), (32, 32, 144, "RN"), (31, 33, 145, "NT"), (65, 36, 400, "CR"),
    (36, 40, 1728, "RT"),
])
def test_no_less_accurate_than_the_fma_chain(products, kind, m, n, k, ops):
    A, B, d = _operands(kind, m, n, k, 7 * m + k)
    sA, sB = (np.ascontiguousarray(_op(x, o)) for x, o in zip((A, B), ops))  # op is its own inverse
    ex = _exact(A, B)
    C = products(ops[0], ops[1], sA, sB, kexp=d)
    e, chain = _err(C, ex), _err(products(ops[0], ops[1], sA, sB, tc=False), ex)
    s = np.ones(k) if d is None else 2.0 ** d
    bound = k * 2.0 ** -55.9 * np.outer(_amax(A / s, 1), _amax(B * s[:, None], 0)) + 2.0 ** -53 * _amax(C[None], 0)
    assert (e <= bound).all()
    # relative to the scale of each entry's row and column, which differ by kind
    w = np.outer(_amax(A / s, 1), _amax(B * s[:, None], 0))
    rms = lambda x: float(np.sqrt(np.mean((x / w) ** 2)))  # noqa: E731
    assert rms(e) <= rms(chain)


def test_scaling_of_k_is_undone_exactly(products):
    """With kneg the scales change sides; a product that needs none keeps its bits under both."""
    A, B, _ = _operands("plain", 33, 40, 50, 1)
    d = np.random.default_rng(0).integers(-20, 20, 50)
    s = 2.0 ** d
    C = products("N", "N", A, B)
    assert np.array_equal(products("N", "N", A * s, B / s[:, None], kexp=d), C)
    assert np.array_equal(products("N", "N", A / s, B * s[:, None], kexp=d, kneg=1), C)


@pytest.mark.parametrize("bits", [0x7FF0000000000000, 0xFFF0000000000000, 0x7FF8000000000000, 0xFFF8000000000000,
                                  0x7FFFFFFFFFFFFFFF, 0xFFFFFFFFFFFFFFFF])
@pytest.mark.parametrize("ops", ["NN", "NT", "TN", "CR"])
def test_non_finite_entries_of_either_sign(products, bits, ops):
    """One such component makes its whole row (column) of C NaN and nothing else."""
    bad = np.array(bits, np.uint64).view(np.float64)
    for side, part in ((0, 0), (0, 1), (1, 0), (1, 1)):
        A, B, d = _operands("plain", 40, 37, 30, 2)
        for scale in (None, np.arange(30) - 15):
            x = (A, B)[side].copy()
            x.view(np.float64).reshape(*x.shape, 2)[5, 7, part] = bad
            args = (x, B) if side == 0 else (A, x)
            sA, sB = (np.ascontiguousarray(_op(y, o)) for y, o in zip(args, ops))
            C = products(ops[0], ops[1], sA, sB, kexp=scale)
            nan = np.isnan(C.real) & np.isnan(C.imag)
            want = np.zeros_like(nan)
            want[(5, slice(None)) if side == 0 else (slice(None), 7)] = True
            assert np.array_equal(nan, want) and np.isfinite(C[~want]).all()
