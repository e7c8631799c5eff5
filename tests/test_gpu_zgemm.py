"""The complex128 tensor-core GEMM (k_ztc.cu) through the calls that use it.

isdf_exchange runs all of its products on it (op N, C and a product of a matrix
with itself, batched over k), with n_p as row, column and inner size; the
reference is the same formula in numpy complex128 from the handle's own X and
V^q.  Sizes sit at the edges of the kernel: 32-row slice blocks, 64 x 32 tiles,
16-k blocks, 384-k chunks, and 96 k where the drain changes its conversion.

Tolerance: with tau = 1e-3 the factor V = L L^H agrees with V_out to
1e-15 / tau = 1e-12 of |V|; sums of n_p <= 400 terms in FP64 keep 1e-13; 1e-10 of
the largest entry leaves two orders of magnitude.
"""
import numpy as np
import pytest

from paper_2601_16379_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cell():
    sh = [W.Shell(0, 0, (0.6,), (1.0,)), W.Shell(0, 1, (0.9,), (1.0,)), W.Shell(1, 1, (1.4,), (1.0,)),
          W.Shell(1, 2, (1.1,), (0.7,))]
    return W.custom_cell(5.0, [[0, 0, 0], [0.37, 0.52, 0.21]], sh, (2, 1, 3), (12, 10, 14))


def _handle(n_p):
    from paper_2601_16379_gb300 import binding as B
    import torch
    cell = _cell()
    g = B.Isdf(cell, B.ISDF_FP64)
    g.set_points(W.seeded_points(cell, n_p, 3))
    g.fit_zeta(1e-3)
    V = torch.empty((cell.nkpts, n_p, n_p), dtype=torch.complex128, device="cuda")
    g.coulomb_metric(V)
    X = g.get(0, torch.empty((cell.nkpts, n_p, cell.nao), dtype=torch.complex128, device="cuda"))
    return cell, g, V, X


def _density(cell):
    rng = np.random.default_rng(5)
    c = rng.standard_normal((cell.nkpts, cell.nao, 4)) + 1j * rng.standard_normal((cell.nkpts, cell.nao, 4))
    return np.einsum("kmi,kni->kmn", c, c.conj())


def _exchange(cell, V, X, P):
    nk = cell.kmesh
    ax = lambda a: np.asarray(a).reshape(*nk, *a.shape[1:])  # noqa: E731
    rho = np.fft.ifftn(ax(X @ P @ X.conj().transpose(0, 2, 1)), axes=(0, 1, 2), norm="forward")
    v = np.fft.fftn(ax(V), axes=(0, 1, 2)).swapaxes(-1, -2)
    g = np.fft.fftn(v * rho, axes=(0, 1, 2)).reshape(V.shape) / cell.nkpts
    return -X.conj().transpose(0, 2, 1) @ g @ X / cell.nkpts


@pytest.mark.parametrize("n_p", [1, 7, 31, 33, 64, 65, 96, 97, 129, 400])
def test_exchange_through_the_tensor_core_gemm(cuda, lib_built, n_p):
    torch = cuda
    cell, g, V, X = _handle(n_p)
    P = _density(cell)
    K = torch.empty((cell.nkpts, cell.nao, cell.nao), dtype=torch.complex128, device="cuda")
    g.exchange(torch.from_numpy(P).cuda(), K)
    ref = _exchange(cell, V.cpu().numpy(), X.cpu().numpy(), P)
    assert np.abs(K.cpu().numpy() - ref).max() <= 1e-10 * np.abs(ref).max()
    g.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e308])
def test_non_finite_input_reaches_the_result(cuda, lib_built, bad):
    """A NaN, an infinity or an overflow in one entry of P spreads over every k of K
    through the convolution, as with FP64 FMAs; nothing finite comes out."""
    torch = cuda
    cell, g, _, _ = _handle(33)
    P = _density(cell)
    P[1, 2, 3] = bad
    K = torch.zeros((cell.nkpts, cell.nao, cell.nao), dtype=torch.complex128, device="cuda")
    g.exchange(torch.from_numpy(P).cuda() * (1e4 if bad == 1e308 else 1.0), K)
    assert not np.isfinite(K.cpu().numpy().view(np.float64)).any()
    g.close()


def test_tiny_and_scaled_inputs(cuda, lib_built):
    """Scaling P by a power of two scales K by it exactly, down to where K is subnormal-free."""
    torch = cuda
    cell, g, _, _ = _handle(65)
    P = torch.from_numpy(_density(cell)).cuda()
    out = []
    for s in (1.0, 2.0 ** -600, 2.0 ** 600):
        K = torch.empty((cell.nkpts, cell.nao, cell.nao), dtype=torch.complex128, device="cuda")
        g.exchange(P * s, K)
        out.append((K / s).cpu().numpy())
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
    g.close()
