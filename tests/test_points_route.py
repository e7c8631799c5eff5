"""Which form of the point selection a cell takes (k_basis.cu, ips_supported), by the library's own symbol: the separable
Gram unless long contractions on few k-points make its terms dearer than a pass over Phi.  The pairs are
measured ones that differ by a tenth or more.
"""
import ctypes as ct
import re
import subprocess

import pytest


class CellDev(ct.Structure):
    _fields_ = [("lat", ct.c_double * 9), ("rec", ct.c_double * 9), ("kmesh", ct.c_int * 3), ("mesh", ct.c_int * 3),
                ("lrange", ct.c_int * 3), ("expcut", ct.c_double), ("orthorhombic", ct.c_int)]


@pytest.mark.parametrize("kmesh,mesh,nao,nterm,separable", [
    ((1, 1, 1), 16, 30, 570, True),        # 3.3 against 4.4 ms
    ((1, 1, 1), 24, 30, 570, True),        # 4.6, 6.0
    ((1, 1, 1), 32, 60, 1140, False),      # 27.7, 21.9
    ((1, 1, 1), 40, 120, 432, True),       # 34, 44
    ((1, 1, 1), 40, 120, 1488, False),     # 79, 44
    ((2, 1, 1), 40, 120, 1488, False),     # 80, 52
    ((2, 2, 2), 40, 120, 1488, True),      # 81, 102
    ((2, 2, 2), 40, 120, 2280, False),     # 116, 103
    ((3, 3, 3), 40, 120, 2280, True),      # 121, 262
    ((1, 1, 1), 16, 8, 8, True),           # no contraction: the terms are the AOs
    ((1, 1, 1), 64, 1024, 1024, True),
    ((10, 10, 10), 24, 26, 26, True),
])
def test_route(lib_built, kmesh, mesh, nao, nterm, separable):
    names = subprocess.run(["nm", "-D", "--defined-only", str(lib_built)], capture_output=True, text=True, check=True).stdout
    fn = getattr(ct.CDLL(str(lib_built)), re.search(r"\b(_ZN4isdf\d+ips_supportedE\w*)", names).group(1))
    fn.restype = ct.c_bool
    c = CellDev(kmesh=kmesh, mesh=(mesh, mesh, mesh), orthorhombic=1)
    assert fn(ct.byref(c), ct.c_int(nterm), ct.c_int(nao)) is separable
    c.orthorhombic = 0
    assert fn(ct.byref(c), ct.c_int(nterm), ct.c_int(nao)) is False
