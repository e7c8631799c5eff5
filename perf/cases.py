"""Performance cases of the k-ISDF fragment-ERI library.

Every case is a call, or a short run of calls, that a program makes through
``paper_2601_16379_gb300.binding.Isdf``.  Sizes are those of the five named
workloads (``workloads.py``), of the GPU tests and of ``bench.py``, with a
smaller real-space grid where the call does not depend on it and the whole
state has to stay small.

The kinds of call:

``points``     interpolation points (Eq. 1, Section II.A); the first thing every program runs
``factor``     least-squares fit and Coulomb metric (Eqs. 2-6) of a k-mesh, V^q kept in the handle, and the
               ERIs of one small fragment through them (V^q itself is no better determined than the
               smallest kept pivot of the fit; the integrals are)
``frag``       fragment ERIs with their J/K traces (Eqs. 17-20) for a batch of fragments
``exchange``   k-point exchange matrix (Eq. 10), once per SCF iteration
``sos``        k-SOS-MP2 polarisability and its trace at one imaginary time (Eqs. 11-15)
``whole``      points, fit, metric and fragments of one small cell in one go
``quartets``   points, fit, metric and AO integrals of a few k-quartets (Eq. 9)

The seed moves the atoms and the lattice constant a little (a geometry of its own
per seed, so no exact symmetry ties), and draws the orbitals, density matrices
and energies.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2601_16379_gb300 import binding as B
from paper_2601_16379_gb300 import workloads as W

PREC = {"fp64": B.ISDF_FP64, "mixed": B.ISDF_MIXED, "fp64tc": B.ISDF_FP64_TC}
SITES = {2: W.BCC2, 4: W.FCC4}
SP = ((0, 0.5), (1, 1.5))                          # c1: (l, exponent) per atom
SPD = ((0, 0.5), (1, 0.5), (1, 1.5), (2, 1.0))     # c2-c5: 13 functions per atom


def _case(name, kind, prec, nk, mesh, n_p, natm=2, basis="spd", a=6.0, tau=1e-7, frags="", quartets=0):
    """nk and mesh are texts "n0 n1 n2"; frags a text of fragment sizes."""
    c = dict(kind=kind, prec=prec, nk=nk, mesh=mesh, n_p=n_p, natm=natm, basis=basis, a=a, tau=tau, frags=frags,
             quartets=quartets)
    return dict(c, name=name) if name else c


def listed():
    return [
        # c1: the smallest cell, everything from the orbitals to the ERIs; launches and host latency
        _case("whole_c1_fp64", "whole", "fp64", "2 2 2", "16 16 16", 64, basis="sp", frags="4"),
        # an anisotropic cell and ragged sizes, as in the parity tests: AO-level integrals of k-quartets
        _case("quartets_ragged_fp64", "quartets", "fp64", "3 2 5", "15 18 20", 150, quartets=3),
        # c5: interpolation points of the paper-scale k-mesh
        _case("points_c5", "points", "mixed", "10 10 10", "24 24 24", 300),
        # c2: fit and metric in plain FP64 at moderate size
        _case("factor_c2_fp64", "factor", "fp64", "3 3 3", "24 24 24", 200, frags="6"),
        # c3: fit and metric of the mixed path, the larger cell and grid
        _case("factor_c3_mixed", "factor", "mixed", "4 4 4", "32 32 32", 500, natm=4, a=7.5, frags="8"),
        # c4: fit and metric of the FP64-class tensor-core path
        _case("factor_c4_fp64tc", "factor", "fp64tc", "6 6 6", "24 24 24", 300, frags="7"),
        # c2: one fragment of 40 orbitals in plain FP64
        _case("frag_c2_fp64", "frag", "fp64", "3 3 3", "16 16 16", 200, frags="40"),
        # c4: uneven fragments in the FP64-class tensor-core path
        _case("frag_c4_fp64tc", "frag", "fp64tc", "6 6 6", "16 16 16", 300, frags="21 40 60 77"),
        # c4: a batch of uneven fragments (sizes of its range, 20 to 120), mixed
        _case("frag_c4_mixed", "frag", "mixed", "6 6 6", "16 16 16", 300,
              frags="23 31 37 42 48 55 61 66 74 83 90 97 105 120"),
        # c5: fragments on the paper-scale k-mesh, mixed
        _case("frag_c5_mixed", "frag", "mixed", "10 10 10", "12 12 12", 300, frags="40 67 100"),
        # c5: exchange matrix of all k
        _case("exchange_c5", "exchange", "fp64", "10 10 10", "12 12 12", 300),
        # c4: polarisability of all Q and the opposite-spin trace at one imaginary time
        _case("sos_c4", "sos", "fp64", "6 6 6", "12 12 12", 300),
    ]


# ----------------------------------------------------------------- sizes
def _ints(s):
    return [int(x) for x in str(s).split()]


def _shells(case):
    return SP if case["basis"] == "sp" else SPD


def _sizes(case):
    nk, mesh = _ints(case["nk"]), _ints(case["mesh"])
    nao = case["natm"] * sum((l + 1) * (l + 2) // 2 for l, _ in _shells(case))
    return math.prod(nk), math.prod(mesh), nao, case["n_p"], _ints(case["frags"])


def work(case):
    """Inputs read once and outputs written once; operations of the method with the
    time-reversal pairing (half of the q) and a factor of rank n_p / 2, about what the
    tolerance of 1e-7 leaves."""
    nk, ng, nao, n_p, frags = _sizes(case)
    kind, r, h = case["kind"], n_p / 2, (nk + 1) / 2
    z = 16.0
    points = dict(bytes=z * nk * nao * (n_p + ng), flops=n_p * n_p * ng + 2.0 * n_p * ng * nao)
    factor = dict(bytes=z * (nk * nao * (n_p + ng) + nk * n_p * n_p),
                  flops=8.0 * h * n_p * ng * nao + 8.0 * h * r * r * ng)
    e = 8.0 if case["prec"] == "mixed" else z
    frag = dict(bytes=sum(z * nk * nao * n + z * n * n + e * n ** 4 for n in frags) + z * nk * n_p * (nao + n_p),
                flops=sum(8.0 * nk * n_p * nao * n + 2.0 * nk * n_p * n * n + 8.0 * n * n * h * r * r
                          + 2.0 * n ** 4 * h * r for n in frags))
    quart = dict(bytes=z * case["quartets"] * nao ** 4, flops=8.0 * case["quartets"] * nao ** 2 * r * (r + nao ** 2))
    if kind == "points":
        parts = [points]
    elif kind == "factor":
        parts = [factor, frag]
    elif kind == "frag":
        parts = [frag]
    elif kind == "whole":
        parts = [points, factor, frag]
    elif kind == "quartets":
        parts = [points, factor, quart]
    elif kind == "exchange":
        parts = [dict(bytes=z * nk * (2 * nao * nao + n_p * nao + n_p * n_p), flops=8.0 * h * (2 * r * r * nao + 2 * r * nao * nao + r ** 3))]
    else:  # sos
        parts = [dict(bytes=z * nk * (nao * nao + n_p * nao + 2 * n_p * n_p), flops=8.0 * h * (n_p * n_p * nao + n_p * nao * nao + 2 * r ** 3))]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def draw(rng):
    """One more case: any of the kinds, meshes cubic or not, sizes odd as well as even."""
    while True:
        kind = rng.choice(["points", "factor", "factor", "frag", "frag", "exchange", "sos", "whole", "quartets"])
        small = kind in ("whole", "quartets")
        prec = "fp64" if small or kind in ("exchange", "sos") else rng.choice(["fp64", "mixed", "fp64tc"])
        if kind == "points":
            prec = "mixed"
        top = 4 if small else 10
        if rng.random() < 0.5:
            nk = [rng.randint(2, top)] * 3
        else:
            nk = [rng.randint(2, top) for _ in range(3)]
        mesh = [rng.randint(10, 20 if kind != "factor" else 32) for _ in range(3)] if rng.random() < 0.6 else [rng.choice([12, 16, 18, 24])] * 3
        natm = rng.choice([2, 2, 4])
        basis = "sp" if small and rng.random() < 0.5 else "spd"
        nao = natm * (4 if basis == "sp" else 13)
        n_p = rng.randint(5 * nao, int(11.5 * nao) if basis == "spd" else 8 * nao)
        a = 6.0 if natm == 2 else 7.5
        frags = ""
        if kind in ("frag", "whole", "factor"):
            count = rng.randint(1, 8) if kind == "frag" else rng.randint(1, 3) if kind == "whole" else 1
            hi = 9 if kind == "factor" else 16 if kind == "whole" else 48 if prec == "fp64" else 72 if prec == "fp64tc" else 120
            frags = " ".join(str(int(round(math.exp(rng.uniform(math.log(3), math.log(hi)))))) for _ in range(count))
        c = _case(None, kind, prec, " ".join(map(str, nk)), " ".join(map(str, mesh)), n_p, natm, basis, a,
                  1e-7, frags, rng.randint(1, 4) if kind == "quartets" else 0)
        k, g, _, _, fr = _sizes(c)
        if k > 1000 or k < 8 or n_p > g // 4:
            continue
        if k in (94, 95, 96, 189, 190, 191, 192) and len(set(nk)) > 1:  # the k-mesh transform refuses these meshes
            continue
        w = work(c)["flops"]
        rows = sum((n * n + 127) // 128 * 128 for n in fr)
        if 16.0 * k * n_p * g > (17e9 if kind == "factor" else 9e9):
            continue
        # the FP64-class path takes fragments of the larger basis in plain FP64
        plain = prec == "fp64" or prec == "fp64tc" and kind == "frag" and natm == 4
        if plain and w > 1.5e11 or w > 2e13 or rows * k * n_p * 20 > 4e10:
            continue
        if kind == "points" and k * nao * g * n_p > 1.1e11:
            continue
        if k * n_p ** 3 > (1.2e10 if kind == "factor" else 2.7e10):
            continue
        return c


# ----------------------------------------------------------------- inputs
def _geometry(case, seed):
    """Lattice constants and atom positions of this seed (orthorhombic cell)."""
    rng = np.random.default_rng([int(seed), 1])
    lat = case["a"] * (1.0 + 0.02 * rng.uniform(-1, 1, 3))
    frac = np.asarray(SITES[case["natm"]], np.float64) + 0.02 * rng.uniform(-1, 1, (case["natm"], 3))
    return lat, frac * lat


def _cell(case, seed):
    lat, coords = _geometry(case, seed)
    shells = [W.Shell(at, l, (x,), (1.0,)) for at in range(case["natm"]) for l, x in _shells(case)]
    return W.Cell(np.diag(lat), coords, shells, tuple(_ints(case["nk"])), tuple(_ints(case["mesh"])))


def _gen(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + tag) & 0x7FFFFFFF)
    return g


def _cgauss(g, *shape):
    return torch.complex(torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64),
                         torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)) * math.sqrt(0.5)


def _isometry(g, n, m):
    """Random n x m matrix with orthonormal columns (n >= m)."""
    x = _cgauss(g, n, m)
    r = torch.linalg.cholesky(x.mH @ x)
    return torch.linalg.solve_triangular(r, x.mH, upper=False).mH.resolve_conj().contiguous()


def _fragments(case, seed):
    nk, _, nao, _, frags = _sizes(case)
    C, gam = [], []
    for i, n in enumerate(frags):
        g = _gen(seed, 10 + i)
        C.append(_isometry(g, nk * nao, n).reshape(nk, nao, n))
        w = _isometry(g, n, max(1, n // 2))
        gamma = 2.0 * (w @ w.mH)
        gam.append((0.5 * (gamma + gamma.mH)).contiguous())
    return C, gam


def _density(case, seed):
    nk, _, nao, _, _ = _sizes(case)
    g = _gen(seed, 3)
    w = torch.linalg.qr(_cgauss(g, nk, nao, nao))[0][:, :, : nao // 4]
    return (2.0 * (w @ w.mH)).contiguous()


def _orbitals(case, seed):
    nk, _, nao, _, _ = _sizes(case)
    C = torch.linalg.qr(_cgauss(_gen(seed, 4), nk, nao, nao))[0].contiguous()
    rng = np.random.default_rng([int(seed), 5])
    n_occ = nao // 4
    occ = np.sort(rng.uniform(-1.0, -0.2, (nk, n_occ)), axis=1)
    vir = np.sort(rng.uniform(0.2, 2.0, (nk, nao - n_occ)), axis=1)
    return C, np.concatenate([occ, vir], axis=1), n_occ


def _quartets(case, seed):
    n = _ints(case["nk"])
    rng = np.random.default_rng([int(seed), 6])
    flat = lambda m: ((m[0] % n[0]) * n[1] + m[1] % n[1]) * n[2] + m[2] % n[2]  # noqa: E731
    out = []
    for _ in range(case["quartets"]):
        k1, k2, k3 = (rng.integers(0, n) for _ in range(3))
        out.append([flat(k1), flat(k2), flat(k3), flat(k3 + k1 - k2)])
    return np.asarray(out, np.int32).reshape(-1, 4)


TAU_IM = 0.6  # imaginary time of the polarisability


def prepare(case, seed):
    nk, ng, nao, n_p, frags = _sizes(case)
    kind = case["kind"]
    empty = lambda *s, dt=torch.complex128: torch.empty(*s, dtype=dt, device="cuda")  # noqa: E731
    s = {"case": case, "seed": int(seed), "h": B.Isdf(_cell(case, seed), PREC[case["prec"]])}
    h = s["h"]
    if kind in ("frag", "whole", "factor"):
        s["C"], s["gamma"] = _fragments(case, seed)
        s["eri"] = [empty(n, n, n, n, dt=torch.complex64 if case["prec"] == "mixed" else torch.complex128) for n in frags]
    if kind == "quartets":
        s["quartets"] = _quartets(case, seed)
        s["out"] = empty(case["quartets"], nao, nao, nao, nao)
    if kind in ("points", "whole"):
        s["X"] = empty(nk, n_p, nao)
    if kind == "exchange":
        s["P"], s["K"] = _density(case, seed), empty(nk, nao, nao)
    if kind == "sos":
        s["C"], s["eps"], s["n_occ"] = _orbitals(case, seed)
        s["chi"] = empty(nk, n_p, n_p)
    if kind in ("factor", "frag", "exchange", "sos"):
        h.build_points(n_p, int(seed))
    if kind in ("frag", "exchange", "sos"):
        h.fit_zeta(case["tau"])
        h.coulomb_metric()
    torch.cuda.synchronize()
    return s


def run(s):
    case, h = s["case"], s["h"]
    kind, n_p, tau = case["kind"], case["n_p"], case["tau"]
    if kind == "points":
        ips = h.build_points(n_p, s["seed"])
        return {"ips": ips, "X": h.get(0, s["X"])}
    if kind == "factor":
        ranks = h.fit_zeta(tau)
        h.coulomb_metric()
        ej, ek = h.fragment_eri(s["C"], s["gamma"], s["eri"])
        return {"ranks": ranks, "ej": ej, "ek": ek, "eri": s["eri"]}
    if kind == "frag":
        ej, ek = h.fragment_eri(s["C"], s["gamma"], s["eri"])
        return {"ej": ej, "ek": ek, "eri": s["eri"]}
    if kind == "exchange":
        return {"K": h.exchange(s["P"], s["K"])}
    if kind == "sos":
        return {"S": h.sos_polarizability(s["C"], s["eps"], s["n_occ"], TAU_IM, s["chi"]), "chi": s["chi"]}
    ips = h.build_points(n_p, s["seed"])
    ranks = h.fit_zeta(tau)
    h.coulomb_metric()
    if kind == "whole":
        ej, ek = h.fragment_eri(s["C"], s["gamma"], s["eri"])
        return {"ips": ips, "ranks": ranks, "ej": ej, "ek": ek, "eri": s["eri"], "X": h.get(0, s["X"])}
    return {"ips": ips, "ranks": ranks, "eri": h.ao_eri(s["quartets"], s["out"])}


# ----------------------------------------------------------------- 64-bit values
def _dfact(n):
    return 1.0 if n < 2 else n * _dfact(n - 2)


def _bloch(case, seed):
    """Phi[k][mu][r] on the grid: per-axis lattice sums of each Cartesian Gaussian."""
    lat, coords = _geometry(case, seed)
    nk, mesh = _ints(case["nk"]), _ints(case["mesh"])
    amin = min(x for _, x in _shells(case))
    phi = []
    for at in range(case["natm"]):
        for l, x in _shells(case):
            for lx in range(l, -1, -1):
                for ly in range(l - lx, -1, -1):
                    lm = (lx, ly, l - lx - ly)
                    norm = math.sqrt((2 * x / math.pi) ** 1.5 * (4 * x) ** l / math.prod(_dfact(2 * v - 1) for v in lm))
                    S = []
                    for ax in range(3):
                        top = math.ceil(math.sqrt(40.0 / amin) / lat[ax]) + 1
                        n = np.arange(-top, top + 1)
                        r = np.arange(mesh[ax]) * lat[ax] / mesh[ax] - coords[at, ax]
                        d = r[None, :] - n[:, None] * lat[ax]
                        ph = np.exp(2j * math.pi * np.outer(np.arange(nk[ax]), n) / nk[ax])
                        S.append(torch.from_numpy(ph @ (d ** lm[ax] * np.exp(-x * d * d))).cuda())
                    phi.append(norm * torch.einsum("ax,by,cz->abcxyz", *S).reshape(math.prod(nk), math.prod(mesh)))
    return torch.stack(phi, 1)


def _splitmix(x):
    m = (1 << 64) - 1
    z = (x + 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _select(phi, n_p, seed):
    """Greedy pivoted Cholesky of the squared Gram matrix, ties by the hash of seed and index."""
    f = phi.reshape(-1, phi.shape[-1])
    f = torch.cat([f.real, f.imag])
    d = f.square().sum(0).square()
    d0 = float(d.max())
    Lt = torch.zeros(n_p, f.shape[1], dtype=torch.float64, device="cuda")
    left = torch.ones_like(d)
    ips = []
    for j in range(n_p):
        m = torch.where(left > 0, d, -torch.inf)
        top = float(m.max())
        cand = (m >= max(top - 1e-11 * d0, 0.5 * top)).nonzero().flatten().tolist()
        p = min(cand, key=lambda r: _splitmix((seed & ((1 << 64) - 1)) ^ r))
        col = (f[:, p] @ f).square() - Lt[:j, p] @ Lt[:j]
        Lt[j] = col / math.sqrt(float(d[p]))
        d -= Lt[j].square()
        left[p] = 0
        ips.append(p)
    return torch.tensor(ips, device="cuda")


def _kfft(x, nk, sign):
    """Unscaled sum over the k-mesh (leading index) with phase exp(sign 2 pi i m.k/n)."""
    y = x.reshape(*nk, -1)
    y = torch.fft.fftn(y, dim=(0, 1, 2)) if sign < 0 else torch.fft.ifftn(y, dim=(0, 1, 2), norm="forward")
    return y.reshape(x.shape)


def _conv(g, nk):
    t = _kfft(g, nk, +1)
    return _kfft((t.real.square() + t.imag.square()).to(torch.complex128), nk, -1) / math.prod(nk)


def _factor_pi(Pi, tau):
    """W[q] with zeta = W^H xi, xi = W eta: inverse of the pivoted Cholesky factor on its pivots."""
    nq, n, _ = Pi.shape
    d = torch.diagonal(Pi, dim1=1, dim2=2).real.clone()
    d0 = d.max(1).values
    L = torch.zeros_like(Pi)
    perm = torch.full((nq, n), -1, dtype=torch.long, device="cuda")
    used = torch.zeros_like(d, dtype=torch.bool)
    alive = torch.ones(nq, dtype=torch.bool, device="cuda")
    rank = torch.zeros(nq, dtype=torch.long, device="cuda")
    at = torch.arange(nq, device="cuda")
    for j in range(n):
        m = torch.where(used, -torch.inf, d)
        top = m.max(1).values
        alive &= (top > tau * d0) & (top > 0)
        if not bool(alive.any()):
            break
        ok = m >= torch.maximum(top - 1e-11 * d0, 0.5 * top)[:, None]
        p = ok.to(torch.int8).argmax(1)
        col = Pi[at, :, p] - (L[:, :, :j] @ L[at, p, :j].conj()[:, :, None])[:, :, 0]
        col = col / torch.sqrt(d[at, p])[:, None]
        col = torch.where(alive[:, None], col, torch.zeros_like(col))
        L[:, :, j] = col
        d -= col.real.square() + col.imag.square()
        used[at[alive], p[alive]] = True
        perm[alive, j] = p[alive]
        rank += alive
    W = torch.zeros_like(Pi)
    for q in range(nq):
        r = int(rank[q])
        s = perm[q, :r]
        inv = torch.linalg.solve_triangular(torch.tril(L[q, s, :r]), torch.eye(r, dtype=L.dtype, device="cuda"), upper=False)
        W[q, :r, :][:, s] = inv
    return W, rank


def _points(case, seed):
    phi = _bloch(case, seed)
    ips = _select(phi, case["n_p"], seed)
    return phi, phi[:, :, ips].transpose(1, 2).contiguous(), ips


def _metric(case, seed, phi, X):
    """Ranks and V^q: the fit and the Coulomb kernel in 64 bits."""
    nk, mesh = _ints(case["nk"]), _ints(case["mesh"])
    K, ng, nao, n_p, _ = _sizes(case)
    lat, _ = _geometry(case, seed)
    Pi = _conv((X.conj() @ X.transpose(1, 2)).contiguous(), nk)
    W, rank = _factor_pi(Pi, case["tau"])
    rx = int(rank.max())
    half = [q for q in range(K) if q <= _minus(q, nk)]
    eta = torch.empty(len(half), n_p, ng, dtype=torch.complex128, device="cuda")
    step = max(1, int(4e9 // (16 * K * ng)))
    for i in range(0, n_p, step):
        eta[:, i:i + step] = _conv((X[:, i:i + step].conj() @ phi).contiguous(), nk)[half]
    V = torch.empty(K, n_p, n_p, dtype=torch.complex128, device="cuda")
    fg = [np.fft.fftfreq(m, 1.0 / m) for m in mesh]
    for i, q in enumerate(half):
        xi = W[q, :rx] @ eta[i]
        m = [q // (nk[1] * nk[2]), (q // nk[2]) % nk[1], q % nk[2]]
        ph = [torch.from_numpy(np.exp(-2j * math.pi * m[a] * np.arange(mesh[a]) / (nk[a] * mesh[a]))).cuda() for a in range(3)]
        c = xi.reshape(rx, *mesh) * torch.einsum("x,y,z->xyz", *ph)
        c = torch.fft.fftn(c, dim=(1, 2, 3)).reshape(rx, ng) / ng
        k = [2 * math.pi / lat[a] * (fg[a] + m[a] / nk[a]) for a in range(3)]
        k2 = (k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2).reshape(-1)
        w = np.where(k2 > 0, 4 * math.pi / np.where(k2 > 0, k2, 1.0), 0.0)
        c = c * torch.from_numpy(np.sqrt(w)).cuda()
        Vx = float(np.prod(lat)) * (c.conj() @ c.transpose(0, 1))
        V[q] = W[q, :rx].transpose(0, 1) @ Vx @ W[q, :rx].conj()
        V[_minus(q, nk)] = V[q].conj() if q != _minus(q, nk) else V[q]
    return V, rank


def _minus(q, nk):
    m = [q // (nk[1] * nk[2]), (q // nk[2]) % nk[1], q % nk[2]]
    return (((-m[0]) % nk[0]) * nk[1] + (-m[1]) % nk[1]) * nk[2] + (-m[2]) % nk[2]


def _eri(case, X, V, C, gamma):
    nk = _ints(case["nk"])
    K, n = X.shape[0], C.shape[-1]
    t = _kfft((X @ C).contiguous(), nk, +1)
    M = (t.conj()[:, :, :, None] * t[:, :, None, :]).reshape(K, X.shape[1], n * n).transpose(1, 2)
    M = _kfft(M.contiguous(), nk, +1) / K
    E = torch.zeros(n * n, n * n, dtype=torch.complex128, device="cuda")
    for q in range(K):
        E += (M[q] @ V[q]) @ M[q].mH
    eri = (E / K).reshape(n, n, n, n).transpose(2, 3).contiguous()
    ej = 0.5 * torch.einsum("pq,rs,pqrs->", gamma, gamma, eri)
    ek = -0.25 * torch.einsum("ps,rq,pqrs->", gamma, gamma, eri)
    return eri, float(ej.real), float(ek.real)


def exact(case, seed):
    nk = _ints(case["nk"])
    K, ng, nao, n_p, frags = _sizes(case)
    kind = case["kind"]
    phi, X, ips = _points(case, seed)
    if kind == "points":
        return {"ips": ips.to(torch.int32), "X": X}
    V, rank = _metric(case, seed, phi, X)
    del phi
    if kind == "exchange":
        P = _density(case, seed)
        rho = _kfft((X @ P @ X.mH).contiguous(), nk, +1)
        G = _kfft(_kfft(V, nk, -1).transpose(1, 2) * rho, nk, -1) / K
        return {"K": -(X.mH @ G @ X) / K}
    if kind == "sos":
        C, eps, n_occ = _orbitals(case, seed)
        Y, w = X @ C, torch.from_numpy(eps).cuda()[:, None, :]
        Yo, Yv = Y[:, :, :n_occ], Y[:, :, n_occ:]
        Go = (Yo * torch.exp(TAU_IM * w[:, :, :n_occ])) @ Yo.mH
        Gv = (Yv * torch.exp(-TAU_IM * w[:, :, n_occ:])) @ Yv.mH
        chi = _kfft(_kfft(Go, nk, +1).transpose(1, 2) * _kfft(Gv, nk, -1), nk, -1) / K
        neg = torch.tensor([_minus(q, nk) for q in range(K)], device="cuda")
        T = V.conj() @ chi @ V.conj()
        return {"S": K * K * float((T * chi[neg]).sum().real), "chi": chi}
    if kind == "quartets":
        out = []
        for k1, k2, k3, k4 in _quartets(case, seed).tolist():
            c = lambda k: np.array([k // (nk[1] * nk[2]), (k // nk[2]) % nk[1], k % nk[2]])  # noqa: E731
            m = (c(k1) - c(k2)) % np.array(nk)
            Q = int((m[0] * nk[1] + m[1]) * nk[2] + m[2])
            a = (X[k1].conj()[:, :, None] * X[k2][:, None, :]).reshape(n_p, -1)
            b = (X[k3].conj()[:, :, None] * X[k4][:, None, :]).reshape(n_p, -1)
            out.append(K * (a.transpose(0, 1) @ V[Q] @ b).reshape(nao, nao, nao, nao))
        return {"ips": ips.to(torch.int32), "ranks": rank.to(torch.int32), "eri": torch.stack(out)}
    C, gamma = _fragments(case, seed)
    eri, ej, ek = [], [], []
    budget = 8e12  # operations that 64 bits do in well under 20 seconds, spent on the smaller fragments first
    for i in sorted(range(len(frags)), key=lambda i: frags[i]):
        n2 = frags[i] ** 2
        budget -= 8.0 * K * n2 * n_p * (n_p + n2)
        eri.append((i, *(_eri(case, X, V, C[i], gamma[i]) if budget > 0 else (None, None, None))))
    eri.sort(key=lambda t: t[0])
    full = all(t[1] is not None for t in eri)
    ej = np.array([t[2] for t in eri]) if full else None
    ek = np.array([t[3] for t in eri]) if full else None
    out = {"ej": ej, "ek": ek, "eri": [t[1] for t in eri]}
    if kind == "whole":
        out |= {"ips": ips.to(torch.int32), "ranks": rank.to(torch.int32), "X": X}
    if kind == "factor":
        out |= {"ranks": rank.to(torch.int32)}
    return out
