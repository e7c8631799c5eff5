"""The complex128 tensor-core products under a small workspace limit (zmul in isdf_api.cu): batch entries
go one at a time, and every entry of the result has the bits it has without the limit.
"""
import numpy as np
import pytest

from paper_2601_16379_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _cell():
    sh = [W.Shell(0, 0, (0.6,), (1.0,)), W.Shell(0, 1, (0.9,), (1.0,)), W.Shell(1, 1, (1.4,), (1.0,)),
          W.Shell(1, 2, (1.1,), (0.7,))]
    return W.custom_cell(5.0, [[0, 0, 0], [0.37, 0.52, 0.21]], sh, (2, 1, 3), (12, 10, 14))


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_same_bits_one_entry_at_a_time(cuda, lib_built, prec):
    from paper_2601_16379_gb300 import binding as B
    torch = cuda
    cell, n_p, out = _cell(), 70, []
    rng = np.random.default_rng(3)
    c = rng.standard_normal((cell.nkpts, cell.nao, 4)) + 1j * rng.standard_normal((cell.nkpts, cell.nao, 4))
    P = torch.from_numpy(np.einsum("kmi,kni->kmn", c, c.conj())).cuda()
    for limit in (None, 1):
        g = B.Isdf(cell, prec)
        if limit:
            g.set_workspace_limit(limit)
        g.set_points(W.seeded_points(cell, n_p, 3))
        g.fit_zeta(1e-6)
        new = lambda *s: torch.empty(s, dtype=torch.complex128, device="cuda")  # noqa: E731
        eta = g.get(2, new(cell.nkpts, n_p, cell.ngrid))
        V = new(cell.nkpts, n_p, n_p)
        g.coulomb_metric(V)
        K = g.exchange(P, new(cell.nkpts, cell.nao, cell.nao))
        out.append([x.cpu().numpy() for x in (eta, V, K)])
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
