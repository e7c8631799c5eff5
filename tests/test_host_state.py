"""Host side of the library (isdf_api.cu) on the CPU, over fakes of the CUDA runtime and the kernels
(host_fakes.cpp): what a handle still offers after an allocation has failed, after a bounded device
wait has expired, and after a new fit.
"""
import ctypes as ct
import subprocess
from pathlib import Path

import numpy as np
import pytest

from paper_2601_16379_gb300 import binding as B
from paper_2601_16379_gb300 import workloads as W

ROOT = Path(__file__).resolve().parents[1]
CSRC = ROOT / "paper_2601_16379_gb300" / "csrc"
CUDA_INCLUDE = "/usr/local/cuda/include"

OOM, TIMEOUT, STATE = -2, -5, -6


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    out = tmp_path_factory.mktemp("host") / "libisdf_host.so"
    inc = ["-I", str(ROOT / "include"), "-I", str(CSRC), "-I", CUDA_INCLUDE]
    subprocess.run(["g++", "-x", "c++", "-std=c++17", "-O1", "-fPIC", "-shared", "-w", "-Wl,-Bsymbolic", *inc,
                    str(CSRC / "isdf_api.cu"), str(ROOT / "tests" / "host_fakes.cpp"), "-o", str(out)], check=True)
    lib = B.load(str(out))
    for f in ("fake_used", "fake_peak", "fake_last_work"):
        getattr(lib, f).restype = ct.c_size_t
    lib.fake_capacity.argtypes = [ct.c_size_t]
    return lib


@pytest.fixture
def fake(fake_lib, monkeypatch):
    monkeypatch.setattr(B, "_lib", fake_lib)
    fake_lib.fake_reset()
    yield fake_lib
    fake_lib.fake_reset()


def _cell(kmesh=(2, 1, 2), mesh=(6, 5, 4)):
    sh = [W.Shell(0, 0, (0.6,), (1.0,)), W.Shell(1, 1, (0.9,), (1.0,))]
    return W.custom_cell(5.0, [[0.01, 0.02, 0.03], [0.37, 0.52, 0.21]], sh, kmesh, mesh)


def _handle(prec=B.ISDF_FP64, n_p=12, **kw):
    g = B.Isdf(_cell(**kw), prec)
    g.set_points(np.arange(n_p))
    return g


def _code(call, *args):
    with pytest.raises(B.IsdfError) as e:
        call(*args)
    return e.value.code


OUT = ct.addressof((ct.c_double * (1 << 16))())  # stands for the caller's buffers, which the fakes do not touch


def test_xi_is_gone_after_its_growth_failed_in_the_eta_route(fake):
    g = _handle()
    g.fit_zeta(1e-3)                     # xi holds 4 of 12 rows
    fake.fake_capacity(fake.fake_used())
    assert _code(g.coulomb_metric_eta) == OOM
    assert _code(g.coulomb_metric) == STATE and _code(g.get, 3, OUT) == STATE
    assert fake.fake_nulls() == 0
    fake.fake_capacity(1 << 40)
    g.coulomb_metric_eta()               # eta still stands
    g.close()


def test_a_fit_that_fails_leaves_no_fit(fake):
    g = _handle()
    g.fit_zeta(1e-3)
    fake.fake_rank(9)                    # a smaller tolerance: more rows of xi
    fake.fake_capacity(fake.fake_used())
    assert _code(g.fit_zeta, 1e-9) == OOM
    assert _code(g.coulomb_metric) == STATE and _code(g.coulomb_metric_eta) == STATE
    assert _code(g.get, 3, OUT) == STATE and fake.fake_nulls() == 0
    fake.fake_capacity(1 << 40)
    g.fit_zeta(1e-9)
    g.coulomb_metric()
    assert fake.fake_nulls() == 0
    g.close()


def test_points_whose_vectors_do_not_fit_leave_no_points(fake):
    g = _handle(n_p=12)
    fake.fake_capacity(fake.fake_used() + 1024)  # the indices fit, X does not
    assert _code(g.set_points, np.arange(40)) == OOM
    assert _code(g.fit_zeta, 1e-3) == STATE and fake.fake_nulls() == 0
    g.close()


@pytest.mark.parametrize("prec", [B.ISDF_FP64, B.ISDF_MIXED, B.ISDF_FP64_TC])
def test_a_fit_that_fails_ends_the_metric_only_once_it_touches_its_factors(fake, prec):
    g = _handle(prec)
    g.fit_zeta(1e-3)
    g.coulomb_metric()
    C = np.zeros((4, 4, 3), np.complex128)
    frag = lambda: g.fragment_eri([_Ptr(C)], traces=False)  # noqa: E731
    frag()
    fake.fake_rank(9)
    fake.fake_capacity(0)
    assert _code(g.fit_zeta, 1e-9) == OOM          # at xi: new pivots beside the old L
    assert _code(frag) == STATE and _code(g.exchange, OUT, OUT) == STATE
    g.close()


def _wide():
    """Eight orbitals: every product of the FP64 fit is long enough for the tensor cores."""
    sh = [W.Shell(a, l, (x,), (1.0,)) for a in (0, 1) for l, x in ((0, 0.6), (1, 0.9))]
    g = B.Isdf(W.custom_cell(5.0, [[0.01, 0.02, 0.03], [0.37, 0.52, 0.21]], sh, (2, 1, 2), (6, 5, 4)), B.ISDF_FP64)
    g.set_points(np.arange(12))
    return g


@pytest.mark.parametrize("product", [0, 1, 2])  # G, g, xi
def test_a_wait_that_expires_in_any_product_fails_the_fit(fake, product):
    g = _wide()
    fake.fake_rank(9)
    fake.fake_arm(product)
    assert _code(g.fit_zeta, 1e-3) == TIMEOUT
    assert _code(g.coulomb_metric) == STATE and _code(g.get, 3, OUT) == STATE
    g.fit_zeta(1e-3)
    assert fake.fake_tc_calls() >= 5
    g.coulomb_metric()
    g.close()


def test_a_call_does_not_report_the_wait_of_one_before(fake):
    g = _wide()
    fake.fake_rank(9)
    g.fit_zeta(1e-3)
    g.coulomb_metric()
    small, large = (_Ptr(np.zeros((4, 8, n), np.complex128)) for n in (3, 64))
    g.fragment_eri([small], traces=False)
    fake.fake_capacity(fake.fake_used())
    fake.fake_arm(0)                                  # in the first fragment; the second does not fit
    assert _code(g.fragment_eri, [small, large]) == OOM
    fake.fake_capacity(1 << 40)
    g.exchange(OUT, OUT)
    g.close()


def _one_entry(slices, m, n, k):
    return (m + n) * ((k + 15) // 16 * 16) * slices * 4 + 256  # zgemm_tc_work_bytes of the fakes, one batch entry


def test_slices_take_what_memory_there_is(fake):
    """g of the FP64_TC fit has one fixed arithmetic: fewer k at a time, never another product."""
    g = _handle(B.ISDF_FP64_TC)                       # n_p = 12, N_g = 120, N_AO = 4, Nk = 4
    g.fit_zeta(1e-3)
    calls = fake.fake_fma_calls(), fake.fake_tc_calls()
    need = fake.fake_used()
    assert fake.fake_last_work() > 3 * _one_entry(7, 12, 120, 4)
    g.close()
    g = _handle(B.ISDF_FP64_TC)
    fake.fake_capacity(need - 2 * _one_entry(7, 12, 120, 4))
    g.fit_zeta(1e-3)
    assert (fake.fake_fma_calls(), fake.fake_tc_calls()) == (2 * calls[0], 2 * calls[1])
    assert fake.fake_last_work() <= 2 * _one_entry(7, 12, 120, 4)
    g.close()


def test_a_product_of_fixed_arithmetic_without_memory_fails(fake):
    g = _handle(B.ISDF_FP64_TC)
    g.fit_zeta(1e-3)
    full = fake.fake_used()
    g.close()
    g = _handle(B.ISDF_FP64_TC)
    base = fake.fake_used()
    # Pi and eta fit, one entry of slices does not
    fake.fake_capacity(base + 16 * 4 * (12 * 12 + 12 * 120) + _one_entry(7, 12, 120, 4) - 1024)
    assert base < full and _code(g.fit_zeta, 1e-3) == OOM
    assert (fake.fake_tc_calls(), fake.fake_fma_calls()) == (1, 3)  # g of the first handle; Pi twice and xi once
    assert _code(g.coulomb_metric) == STATE
    g.close()


def test_slices_keep_to_the_workspace_limit(fake):
    g = _handle(B.ISDF_FP64_TC)
    g.lib.isdf_set_workspace_limit(g.h, 1)
    g.fit_zeta(1e-3)
    assert fake.fake_last_work() == _one_entry(7, 12, 120, 4)
    g.close()


def test_slices_give_way_to_what_is_allocated_later(fake):
    """What held without slices holds with them: the metric needs every byte."""
    g = _wide()
    fake.fake_rank(9)
    g.fit_zeta(1e-3)
    g.coulomb_metric()
    g.close()
    g = _wide()
    g.fit_zeta(1e-3)
    # V_xi is there; LtV, L and the small arrays of the metric follow
    fake.fake_capacity(fake.fake_used() + 2 * 16 * 4 * 12 * 12)
    g.coulomb_metric()
    assert fake.fake_nulls() == 0
    g.close()


@pytest.mark.parametrize("room", [True, False])
def test_slices_free_the_other_group_only_if_that_is_enough(fake, room):
    """E = B B^H of an FP64 fragment without memory for its slices: with eta and xi gone they fit (room), and the
    documented price is a new fit; else the product runs as FMA chains and eta stays."""
    g = _wide()
    fake.fake_rank(9)
    g.fit_zeta(1e-3)
    g.coulomb_metric()
    C = _Ptr(np.zeros((4, 8, 24), np.complex128))
    g.fragment_eri([C], traces=False)
    fma, used = fake.fake_fma_calls(), fake.fake_used()
    g.close()
    g = _wide()
    g.fit_zeta(1e-3)
    g.coulomb_metric()
    # B = M L keeps one q at a time; E needs 864 KB, eta and xi hold 154
    free = 840 if room else 600
    fake.fake_capacity(used - 4 * _one_entry(8, 24 * 24, 12, 12) + (free << 10))
    base = fake.fake_fma_calls()
    g.fragment_eri([C], traces=False)
    assert fma == base and fake.fake_fma_calls() == base + (0 if room else 1)
    fake.fake_capacity(1 << 40)
    if room:
        assert _code(g.coulomb_metric_eta) == STATE
    else:
        g.coulomb_metric_eta()
    g.close()


def test_products_with_w_scale_their_inner_index(fake):
    """L = W^T L_xi and the two products of V_out: rows of W and of the other operand are graded against each other."""
    g = _wide()
    fake.fake_rank(9)
    g.fit_zeta(1e-3)
    g.coulomb_metric(OUT)
    assert fake.fake_kexp_calls() == 3
    g.close()


@pytest.mark.parametrize("rank", [40, 80, 96])
def test_b_of_mixed_fragments_takes_the_place_of_z(fake, rank):
    """Z and M as wide as the points hold M and B of any rank; only at full rank B is the larger of Z and B, by the
    q of the sum beyond half of the mesh (70 of 120 here)."""
    kmesh, n_p, nf = (6, 4, 5), 96, 40
    g = _handle(B.ISDF_MIXED, n_p=n_p, kmesh=kmesh, mesh=(5, 5, 5))
    g.lib.isdf_set_workspace_limit(g.h, 1)
    fake.fake_rank(rank)
    g.fit_zeta(1e-3)
    g.coulomb_metric()
    base = fake.fake_used()
    nk, n_s, rows = 120, 70, nf * nf
    g.fragment_eri([_Ptr(np.zeros((nk, 4, nf), np.complex128))], traces=False)
    z, m, b = 4 * nk * rows * n_p, 8 * n_s * rows * n_p, 8 * n_s * rows * rank
    rest = 8 * nk * n_p * nf + 16 * rows * n_p        # T, one q of slices, maps and row maxima
    assert fake.fake_peak() - base <= max(z, b) + m + rest
    g.close()


class _Ptr:
    def __init__(self, a):
        self.a, self.shape = a, a.shape

    def data_ptr(self):
        return self.a.ctypes.data
