"""What is measured of this library: the calls that a QS^3 program makes, over
the sizes the library is used at.

A case names one public entry point, a lattice, a number of down spins, the
momentum sectors and the vector type.  The listed cases are the workloads of
the repository's own configurations, tests and benchmark (the 16-site chain,
the 10x10 square lattice with its momentum sectors, the 6x6x6, 8x8x8 and
10x10x10 cubes, the bond-disordered open square lattice); draw() varies the
lattice, its sides, N_down, the sectors and the type around them.

exact() restates each result from its definition with plain torch in 64 bits:
states as sorted site lists, ranks by the combinatorial number system, orbit
minima over every translation.  It uses nothing of the library.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2107_00872_gb300 as qs3

DEV = "cuda"
REAL = {"f32": torch.float32, "f64": torch.float64, "c64": torch.float32, "c128": torch.float64}


# ---------------------------------------------------------------- the cases

def listed() -> list:
    return [
        # the smallest call: one product on the 16-site chain (560 states),
        # where launch latency is all there is
        dict(name="chain16_hphi_f64", kind="hphi", geom="chain", lx=16, ly=1, lz=1, nd=3, k="none", dtype="f64"),
        # the largest: the bond-disordered open 32x32 lattice without
        # symmetry, 178,433,024 states, fp32 vectors (the bulk product of a
        # mixed-precision ground-state run)
        dict(name="open32_hphi_f32", kind="hphi", geom="open", lx=32, ly=32, lz=1, nd=3, k="none", dtype="f32"),
        # the same model in binary64 at an ordinary size (31,628,736 states)
        dict(name="open24_hphi_f64", kind="hphi", geom="open", lx=24, ly=24, lz=1, nd=3, k="none", dtype="f64"),
        # all 100 momentum sectors of the 10x10 lattice in one product:
        # complex128 arithmetic, and the product on the integer units
        dict(name="square10_allk_hphi_c128", kind="hphi", geom="square", lx=10, ly=10, lz=1, nd=4, k="all",
             dtype="c128"),
        dict(name="square10_allk_hphi_int", kind="hphi", geom="square", lx=10, ly=10, lz=1, nd=4, k="all",
             dtype="c128", integer=True),
        # sectors too large for a representative table: the 6x6x6 cube with
        # five down spins at k = 0 (17,313,563 representatives), and the
        # 8x8x8 cube with four in fp32
        dict(name="cubic6_nd5_gamma_hphi_c128", kind="hphi", geom="cubic", lx=6, ly=6, lz=6, nd=5, k="gamma",
             dtype="c128"),
        dict(name="cubic8_nd4_gamma_hphi_c64", kind="hphi", geom="cubic", lx=8, ly=8, lz=8, nd=4, k="gamma",
             dtype="c64"),
        # S^-_q applied to a four-spin state: the start of a dynamical
        # structure factor (about 752,900 target rows per q)
        dict(name="square10_smq", kind="smq", geom="square", lx=10, ly=10, lz=1, nd=4, k="some", nk=1, kseed=3,
             dtype="c128"),
        # two-point functions and S(q) at every q of a state of one sector
        dict(name="square10_correlations", kind="corr", geom="square", lx=10, ly=10, lz=1, nd=4, k="gamma",
             dtype="c128"),
        # setting a problem up: the basis of all momenta from the lattice,
        # and the first product on it
        dict(name="square10_allk_setup", kind="setup", geom="square", lx=10, ly=10, lz=1, nd=4, k="all",
             dtype="c128"),
        # whole calls: the ground states of all 100 sectors at once, and the
        # smallest problem from start to end (ground state of the 16-site
        # chain, then every two-point function)
        dict(name="square10_allk_lanczos", kind="lanczos", geom="square", lx=10, ly=10, lz=1, nd=4, k="all",
             dtype="c128", n_max=250),
        dict(name="chain16_ground_state", kind="ground", geom="chain", lx=16, ly=1, lz=1, nd=3, k="none",
             dtype="f64", n_max=160),
    ]


def draw(rng: random.Random) -> dict:
    """One more case of the listed ranges (no name)."""
    while True:
        c = _draw(rng)
        if _fits(c):
            return c


def _log(rng, lo, hi) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng) -> dict:
    kind = rng.choice(["hphi_u1", "hphi_u1", "hphi_k", "hphi_k", "hphi_search", "smq", "corr", "setup", "lanczos",
                       "ground"])
    c = dict(kind=kind, lx=1, ly=1, lz=1)
    some = dict(k="some", nk=_log(rng, 1, 24), kseed=rng.randrange(1 << 30))
    if kind == "hphi_u1":
        if rng.random() < 0.4:
            c.update(geom="chain", lx=_log(rng, 12, 64))
        else:
            c.update(geom="open", lx=_log(rng, 5, 32))
            c.update(ly=max(3, c["lx"] - rng.randrange(4)))
        c.update(kind="hphi", nd=rng.choice([2, 3, 3, 3, 4]), k="none", dtype=rng.choice(["f32", "f64"]))
        return c
    if kind == "hphi_search":
        # sectors beyond the representative table
        lx = rng.choice([5, 6, 7, 8])
        c.update(kind="hphi", geom="cubic", lx=lx, ly=lx - rng.randrange(2), lz=lx, nd=rng.choice([4, 5]), k="some",
                 nk=rng.choice([1, 1, 2]), kseed=rng.randrange(1 << 30), dtype=rng.choice(["c64", "c128"]))
        return c
    if kind == "hphi_k":
        if rng.random() < 0.75:
            c.update(geom="square", lx=rng.randrange(4, 13), ly=rng.randrange(4, 13))
        else:
            c.update(geom="cubic", lx=rng.randrange(3, 8), ly=rng.randrange(3, 8), lz=rng.randrange(3, 8))
        c.update(kind="hphi", nd=rng.choice([2, 3, 3, 4, 4]), dtype=rng.choice(["c64", "c128", "c128"]))
        c.update(rng.choice([dict(k="all"), some]))
        if c["dtype"] == "c128" and rng.random() < 0.5:
            c["integer"] = True
        return c
    if kind in ("smq", "corr"):
        c.update(geom="square", lx=rng.randrange(4, 11), ly=rng.randrange(4, 11), nd=rng.choice([2, 3, 4]), k="some",
                 nk=1, kseed=rng.randrange(1 << 30), dtype="c128")
        return c
    if kind == "setup":
        if rng.random() < 0.7:
            c.update(geom="square", lx=rng.randrange(5, 11), ly=rng.randrange(5, 11))
        else:
            c.update(geom="cubic", lx=rng.randrange(4, 7), ly=rng.randrange(4, 7), lz=rng.randrange(4, 7))
        c.update(nd=rng.choice([3, 4]), dtype="c128")
        c.update(rng.choice([dict(k="all"), some]))
        return c
    if kind == "lanczos":
        c.update(geom="square", lx=rng.randrange(5, 11), ly=rng.randrange(5, 11), nd=rng.choice([3, 4]), dtype="c128",
                 n_max=250)
        c.update(rng.choice([dict(k="all"), some]))
        return c
    c.update(geom="chain", lx=_log(rng, 12, 40), nd=rng.choice([2, 3, 4]), k="none", dtype="f64", n_max=160)
    return c


def _sites(c) -> int:
    return c["lx"] * c["ly"] * c["lz"]


def _rows(c) -> float:
    """The number of rows, exact without momenta, else C(N, N_down) / N per sector."""
    n = _sites(c)
    if c["k"] == "none":
        return float(math.comb(n, c["nd"]))
    s = {"all": n, "gamma": 1}.get(c["k"], min(c.get("nk", 1), n))
    return math.comb(n, c["nd"]) / n * s


def _fits(c) -> bool:
    """Whether a drawn case stays within the listed ranges."""
    n, states = _sites(c), math.comb(_sites(c), c["nd"])
    if n < 2 * c["nd"] or min(v for v in (c["lx"], c["ly"], c["lz"]) if v > 1) < 3:
        return False
    r = _rows(c)
    if c["kind"] == "hphi":
        if c["k"] == "none":
            return 500 <= r <= (1.79e8 if c["dtype"] == "f32" else 3.2e7)
        if c.get("integer"):
            # within the representative table
            return r >= 500 and r <= 4e6 and states * 4 + states / n * 4 * n < 5e8 and states / n < 1e6
        return 500 <= r <= (1.8e7 if states > 2.7e8 else 4e6)
    if c["kind"] == "smq":
        return states / n >= 20 and math.comb(n, c["nd"] + 1) / n <= 8e5
    if c["kind"] == "ground":
        return 200 <= r <= 1e5
    return 100 <= r <= 4e6


# ------------------------------------------------------------------ lattices

def _dims(c):
    return (c["lx"], c["ly"], c["lz"])


def _lattice(c, seed):
    """Nearest-neighbour bonds of the case's lattice, site r = x + Lx (y + Ly
    z).  "open": open boundaries with J ~ U[0.5, 1.5], Jz = 0.8 J and fields
    h ~ U[-0.1, 0.1] from the seed; else periodic with J = 1 and one
    anisotropy Jz ~ U[0.9, 1.1] from the seed (the ground-state cases: Jz = 1)."""
    lx, ly, lz = dims = _dims(c)
    periodic = c["geom"] != "open"
    bi, bj = [], []
    for z in range(lz):
        for y in range(ly):
            for x in range(lx):
                r = x + lx * (y + ly * z)
                for a, d in enumerate(((1, 0, 0), (0, 1, 0), (0, 0, 1))):
                    if dims[a] == 1:
                        continue
                    p = [x + d[0], y + d[1], z + d[2]]
                    if p[a] >= dims[a]:
                        if not periodic:
                            continue
                        p[a] = 0
                    bi.append(r)
                    bj.append(p[0] + lx * (p[1] + ly * p[2]))
    rng = np.random.default_rng(seed)
    nb, n = len(bi), lx * ly * lz
    h = None
    if periodic:
        jxy = np.ones(nb)
        jz = np.full(nb, 1.0 if c["kind"] in ("lanczos", "ground") else rng.uniform(0.9, 1.1))
    else:
        jxy = rng.uniform(0.5, 1.5, nb)
        jz = 0.8 * jxy
        h = rng.uniform(-0.1, 0.1, n)
    return SimpleNamespace(n_sites=n, bi=np.array(bi, np.int32), bj=np.array(bj, np.int32), jxy=jxy, jz=jz, h=h,
                           L=dims if periodic else (0, 0, 0), pos=None, n_sub=1)


def _momenta(c):
    """The momenta of the case's sectors (None: no translation symmetry)."""
    lx, ly, lz = _dims(c)
    if c["k"] == "none":
        return None
    if c["k"] == "gamma":
        return [(0, 0, 0)]
    ks = [(x, y, z) for z in range(lz) for y in range(ly) for x in range(lx)]
    if c["k"] == "all":
        return ks
    random.Random(c["kseed"]).shuffle(ks)
    return ks[:c["nk"]]


def _transfer(c):
    """The momentum transfer of S^-_q, and the target momentum."""
    lx, ly, lz = _dims(c)
    r = random.Random(c["kseed"] + 1)
    q = (r.randrange(lx), r.randrange(ly), r.randrange(lz))
    k = _momenta(c)[0]
    return q, tuple((k[a] + q[a]) % _dims(c)[a] for a in range(3))


def _grid_q(c):
    """Every wave vector of the lattice, q.a_alpha in radians."""
    lx, ly, lz = _dims(c)
    return np.array([(2 * np.pi * x / lx, 2 * np.pi * y / ly, 2 * np.pi * z / lz)
                     for z in range(lz) for y in range(ly) for x in range(lx)])


def _vector(c, n, seed):
    """A normalised Gaussian vector, as Lanczos vectors are."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    cplx = c["dtype"][0] == "c"
    v = torch.randn(n * (2 if cplx else 1), generator=g, device=DEV, dtype=REAL[c["dtype"]])
    v /= torch.linalg.vector_norm(v, dtype=torch.float64).to(v.dtype)
    return torch.view_as_complex(v.view(n, 2)) if cplx else v


# ------------------------------------------------------------- prepare, run

def prepare(case, seed) -> dict:
    c = dict(case)
    lat, ks = _lattice(c, seed), _momenta(c)
    st = dict(case=c, lattice=lat, ks=ks)
    basis = qs3.Basis(lat, c["nd"], ks)
    if c["kind"] == "setup":
        # the vector a program would have in hand; the basis is built anew in each pass
        st["phi"] = _vector(c, basis.total_dim, seed)
        basis.close()
        return st
    st["basis"] = basis
    if c["kind"] in ("lanczos", "ground"):
        st["opts"] = qs3.SolveOpts(n_max=c["n_max"], min_iter=20, check_every=5, eps=1e-14, res_tol=1e-12,
                                   seed=int(seed) + 1)
        st["pairs"] = [(i, j) for i in range(lat.n_sites) for j in range(lat.n_sites)]
        return st
    st["phi"] = _vector(c, basis.total_dim, seed)
    if c["kind"] == "smq":
        st["q"], kq = _transfer(c)
        st["target"] = qs3.Basis(lat, c["nd"] + 1, [kq])
    if c["kind"] == "corr":
        st["pairs"] = [(0, j) for j in range(lat.n_sites)]
        st["qs"] = _grid_q(c)
    return st


def run(st):
    c, phi = st["case"], st.get("phi")
    kind = c["kind"]
    if kind == "hphi":
        return st["basis"].hphi(phi, integer=bool(c.get("integer")))
    if kind == "smq":
        return qs3.smq(st["basis"], 0, phi, st["target"], 0, st["q"])
    if kind == "corr":
        return st["basis"].correlations(phi, 0, pairs=st["pairs"], q=st["qs"], local=True)
    if kind == "setup":
        basis = qs3.Basis(st["lattice"], c["nd"], st["ks"])
        return {"dims": np.array(basis.dims), "psi": basis.hphi(phi)}
    ev, vec, _ = st["basis"].lanczos(st["opts"], vectors=True)
    if kind == "lanczos":
        return {"e": ev, "v": vec}
    return {"e": ev, "v": vec, "corr": st["basis"].correlations(vec, 0, pairs=st["pairs"], local=True)}


# --------------------------------------------------------------------- work

def work(case) -> dict:
    """Bytes and operations of one pass: every input vector read once, every
    output written once; a product of 2 (real) or 8 (complex) operations per
    off-diagonal term."""
    c = dict(case)
    n, nd, d = _sites(c), c["nd"], _rows(c)
    cplx = c["dtype"][0] == "c"
    size = REAL[c["dtype"]].itemsize * (2 if cplx else 1)
    deg = 2 * sum(1 for v in _dims(c) if v > 1)
    terms = d * nd * deg
    hphi = {"bytes": 2 * size * d, "flops": terms * (8 if cplx else 2)}
    kind = c["kind"]
    if kind == "hphi" or kind == "setup":
        return hphi
    if kind == "smq":
        t = math.comb(n, nd + 1) / n
        return {"bytes": size * (d + t), "flops": 8 * t * (nd + 1)}
    if kind == "corr":
        return {"bytes": size * d, "flops": 8 * d * nd * (n - nd)}
    # Lanczos: a nominal number of steps, each one product and one pass over
    # the Krylov basis of so many vectors
    steps = min(100.0 if kind == "lanczos" else 60.0, d)
    w = {"bytes": steps * hphi["bytes"] + size * d * steps * steps / 2,
         "flops": steps * hphi["flops"] + (16 if cplx else 4) * d * steps * steps / 2}
    if kind == "ground":
        w["flops"] += 2 * d * nd * (n - nd)
    return w


# -------------------------------------------------------------------- exact

def _binom(n, m):
    """C(x, m) for x = 0 .. n as a 64-bit tensor."""
    return torch.tensor([math.comb(x, m) for x in range(n + 1)], dtype=torch.int64, device=DEV)


def _states(ranks, n, nd):
    """Ascending site lists [len, nd] of the ranks sum_m C(c_m, m + 1)."""
    r, cols = ranks.clone(), []
    for m in range(nd, 0, -1):
        t = _binom(n, m)
        x = torch.searchsorted(t, r, right=True) - 1
        cols.append(x)
        r -= t[x]
    return torch.stack(cols[::-1], 1)


def _rank(c, n):
    """The ranks of ascending site lists."""
    return sum(_binom(n, m + 1)[c[:, m]] for m in range(c.shape[1]))


def _adjacency(lat):
    """Neighbour, hop amplitude J / 2 and Jz per site, padded with itself and zeros."""
    nbr = [[] for _ in range(lat.n_sites)]
    for i, j, x, z in zip(lat.bi.tolist(), lat.bj.tolist(), lat.jxy.tolist(), lat.jz.tolist()):
        nbr[i].append((j, x / 2, z))
        nbr[j].append((i, x / 2, z))
    w = max(len(v) for v in nbr)
    t = [[v[b] if b < len(v) else (i, 0.0, 0.0) for b in range(w)] for i, v in enumerate(nbr)]
    col = lambda k, dt: torch.tensor([[e[k] for e in v] for v in t], dtype=dt, device=DEV)  # noqa: E731
    return col(0, torch.int64), col(1, torch.float64), col(2, torch.float64)


def _diagonal(c, lat, nbr, jz):
    """sum_b Jz s^z s^z - sum_i h_i s^z_i of the states c."""
    h = torch.zeros(lat.n_sites, dtype=torch.float64, device=DEV)
    if lat.h is not None:
        h = torch.tensor(lat.h, dtype=torch.float64, device=DEV)
    d = torch.full((c.shape[0],), float(lat.jz.sum()) / 4 - float(h.sum()) / 2, dtype=torch.float64, device=DEV)
    site = -jz.sum(1) / 2 + h
    for m in range(c.shape[1]):
        d += site[c[:, m]]
        for b in range(nbr.shape[1]):
            j = nbr[c[:, m], b]
            d += 0.5 * jz[c[:, m], b] * (c == j[:, None]).any(1)
    return d


def _hops(c, nbr, amp):
    """For each spin and neighbour: (the moved site lists, amplitude, whether the move is one)."""
    for m in range(c.shape[1]):
        for b in range(nbr.shape[1]):
            j = nbr[c[:, m], b]
            ok = ~(c == j[:, None]).any(1)
            t = c.clone()
            t[:, m] = torch.where(ok, j, c[:, m])
            yield torch.sort(t, 1).values, amp[c[:, m], b], ok


def _hphi_u1(lat, nd, phi):
    n = lat.n_sites
    nbr, amp, jz = _adjacency(lat)
    x = phi.to(torch.float64)
    out = torch.empty_like(x)
    step = 1 << 23
    for r0 in range(0, x.numel(), step):
        r = torch.arange(r0, min(r0 + step, x.numel()), device=DEV)
        c = _states(r, n, nd)
        acc = _diagonal(c, lat, nbr, jz) * x[r]
        for t, a, ok in _hops(c, nbr, amp):
            acc += torch.where(ok, a * x[_rank(t, n)], 0.0)
        out[r] = acc
    return out


def _translations(c, dims):
    """Every translation u of the lists c: (u, the sorted lists moved by -u)."""
    lx, ly, lz = dims
    x, y, z = c % lx, (c // lx) % ly, c // (lx * ly)
    for u in range(lx * ly * lz):
        ux, uy, uz = u % lx, (u // lx) % ly, u // (lx * ly)
        t = (x - ux) % lx + lx * ((y - uy) % ly + ly * ((z - uz) % lz))
        yield u, torch.sort(t, 1).values


def _canon(c, dims):
    """(rank of the representative, translation u with c = T_u rep) of each list."""
    n = dims[0] * dims[1] * dims[2]
    best = torch.full((c.shape[0],), 1 << 62, dtype=torch.int64, device=DEV)
    at = torch.zeros_like(best)
    for u, t in _translations(c, dims):
        r = _rank(t, n)
        less = r < best
        best = torch.where(less, r, best)
        at = torch.where(less, u, at)
    return best, at


def _orbits(n, nd, dims):
    """Sorted ranks of every orbit's representative, from the lists that hold site 0."""
    rest = _states(torch.arange(math.comb(n - 1, nd - 1), device=DEV), n - 1, nd - 1) + 1 if nd > 1 else None
    c = torch.zeros((1, 1), dtype=torch.int64, device=DEV) if nd == 1 else torch.cat(
        [torch.zeros((rest.shape[0], 1), dtype=torch.int64, device=DEV), rest], 1)
    reps = torch.unique(_canon(c, dims)[0])
    return reps


def _phase(k, u, dims):
    """e^{-2 pi i k.u / L} of translations u (flat site indices)."""
    lx, ly, lz = dims
    n = lx * ly * lz
    num = (k[0] * (u % lx) * (n // lx) + k[1] * ((u // lx) % ly) * (n // ly) + k[2] * (u // (lx * ly)) * (n // lz)) % n
    a = -2.0 * math.pi * num.to(torch.float64) / n
    return torch.complex(torch.cos(a), torch.sin(a))


class _Sectors:
    """The orbits of a lattice and, per momentum, its rows."""

    def __init__(self, n, nd, dims, ks):
        self.n, self.nd, self.dims = n, nd, dims
        self.reps = _orbits(n, nd, dims)
        self.lists = _states(self.reps, n, nd)
        self.stab = torch.zeros_like(self.reps)
        bad = torch.zeros((len(ks), self.reps.numel()), dtype=torch.bool, device=DEV)
        for u, t in _translations(self.lists, dims):
            fix = _rank(t, n) == self.reps
            self.stab += fix
            for s, k in enumerate(ks):
                num = (k[0] * (u % dims[0]) * (n // dims[0]) + k[1] * ((u // dims[0]) % dims[1]) * (n // dims[1]) +
                       k[2] * (u // (dims[0] * dims[1])) * (n // dims[2])) % n
                if num:
                    bad[s] |= fix
        self.members = [torch.nonzero(~bad[s])[:, 0] for s in range(len(ks))]
        self.rows = []
        for m in self.members:
            r = torch.full_like(self.reps, -1)
            r[m] = torch.arange(m.numel(), device=DEV)
            self.rows.append(r)

    def find(self, c):
        """(orbit, translation) of each list."""
        r, u = _canon(c, self.dims)
        return torch.searchsorted(self.reps, r), u


def _hphi_k(c, lat, ks, phi):
    n, nd, dims = lat.n_sites, c["nd"], _dims(c)
    sec = _Sectors(n, nd, dims, ks)
    nbr, amp, jz = _adjacency(lat)
    x = phi.to(torch.complex128)
    diag = _diagonal(sec.lists, lat, nbr, jz)
    hops = [(*sec.find(t), a, ok) for t, a, ok in _hops(sec.lists, nbr, amp)]
    out, off = torch.empty_like(x), 0
    for s, k in enumerate(ks):
        mem, rows = sec.members[s], sec.rows[s]
        d = mem.numel()
        v = x[off:off + d]
        acc = diag[mem] * v
        for g, u, a, ok in hops:
            g, u, a, ok = g[mem], u[mem], a[mem], ok[mem]
            r = rows[g]
            ok = ok & (r >= 0)
            w = a * torch.sqrt(sec.stab[g].to(torch.float64) / sec.stab[mem].to(torch.float64))
            acc += torch.where(ok, w * _phase(k, u, dims) * v[r.clamp(min=0)], 0.0)
        out[off:off + d] = acc
        off += d
    return out, np.array([m.numel() for m in sec.members])


def _smq(c, lat, phi, q, k, kq):
    n, nd, dims = lat.n_sites, c["nd"], _dims(c)
    src, dst = _Sectors(n, nd, dims, [k]), _Sectors(n, nd + 1, dims, [kq])
    mem = dst.members[0]
    lists, stab = dst.lists[mem], dst.stab[mem].to(torch.float64)
    acc = torch.zeros(mem.numel(), dtype=torch.complex128, device=DEV)
    for m in range(nd + 1):
        g, u = src.find(torch.cat([lists[:, :m], lists[:, m + 1:]], 1))
        r = src.rows[0][g]
        w = torch.sqrt(src.stab[g].to(torch.float64) / stab) * _phase(k, u, dims) * _phase(q, lists[:, m], dims)
        acc += torch.where(r >= 0, w * phi[r.clamp(min=0)], 0.0)
    return acc / math.sqrt(n)


def _disp(a, b, dims):
    """Displacement b - a of site indices."""
    lx, ly, lz = dims
    return (b % lx - a % lx) % lx + lx * (((b // lx) % ly - (a // lx) % ly) % ly + ly * ((b // (lx * ly) - a // (lx * ly)) % lz))


def _corr_k(c, lat, k, phi, pairs, qs):
    n, nd, dims = lat.n_sites, c["nd"], _dims(c)
    sec = _Sectors(n, nd, dims, [k])
    mem = sec.members[0]
    lists, stab = sec.lists[mem], sec.stab[mem].to(torch.float64)
    w = (phi.conj() * phi).real
    zz = torch.zeros(n, dtype=torch.float64, device=DEV)
    for a in range(nd):
        for b in range(nd):
            zz.index_add_(0, _disp(lists[:, a], lists[:, b], dims), w)
    pm = torch.zeros(n, dtype=torch.complex128, device=DEV)
    for m in range(nd):
        for j in range(n):
            ok = ~(lists == j).any(1)
            t, x, l, s = lists[ok].clone(), phi[ok], lists[ok], stab[ok]
            t[:, m] = j
            g, u = sec.find(torch.sort(t, 1).values)
            r = sec.rows[0][g]
            f = torch.sqrt(sec.stab[g].to(torch.float64) / s) / n * _phase(k, u, dims) * phi[r.clamp(min=0)]
            f = torch.where(r >= 0, x.conj() * f, 0.0)
            d = _disp(torch.full_like(l[:, m], j), l[:, m], dims)
            pm.index_add_(0, d, f)
    norm = float(w.sum())
    zz, pm = (zz / (n * norm)).cpu().numpy() + 0.25 - nd / n, (pm / norm).cpu().numpy()
    zz[0], pm[0] = 0.25, 1.0 - nd / n
    out = {"szsz": np.array([zz[_disp(i, j, dims)] for i, j in pairs]),
           "spsm": np.array([pm[_disp(i, j, dims)] for i, j in pairs]), "sz": np.full(n, 0.5 - nd / n)}
    site = np.arange(n)
    pos = np.stack([site % dims[0], (site // dims[0]) % dims[1], site // (dims[0] * dims[1])], 1)
    dd = _disp(site[:, None], site[None, :], dims)          # displacement r' - r
    e = np.exp(1j * qs @ pos.T)
    f = e[:, :, None] * e[:, None, :].conj()
    out["sq_zz"] = (f * zz[dd]).sum((1, 2)).real / n
    out["sq_pm"] = (f * pm[dd]).sum((1, 2)).real / n
    return out


def _ground(c, lat, pairs):
    """The lowest level by dense diagonalisation and its two-point functions
    (the vector's sign is free: no value)."""
    n, nd = lat.n_sites, c["nd"]
    d = math.comb(n, nd)
    nbr, amp, jz = _adjacency(lat)
    s = _states(torch.arange(d, device=DEV), n, nd)
    h = torch.diag(_diagonal(s, lat, nbr, jz))
    i = torch.arange(d, device=DEV)
    for t, a, ok in _hops(s, nbr, amp):
        h[i[ok], _rank(t, n)[ok]] += a[ok]
    ev, vec = np.linalg.eigh(h.cpu().numpy())
    if ev[1] - ev[0] < 1e-8:
        return {"e": ev[:1].reshape(1, 1), "v": None, "corr": {"szsz": None, "spsm": None, "sz": None}}
    v = torch.tensor(vec[:, 0].copy(), device=DEV)
    occ = torch.zeros((d, n), dtype=torch.float64, device=DEV).scatter_(1, s, 1.0)
    sz = 0.5 - occ
    zz = (sz * (v * v)[:, None]).T @ sz
    pm = torch.zeros((n, n), dtype=torch.float64, device=DEV)
    for m in range(nd):
        for j in range(n):
            ok = ~(s == j).any(1)
            t = s[ok].clone()
            t[:, m] = j
            pm.view(-1).index_add_(0, s[ok][:, m] * n + j, v[_rank(torch.sort(t, 1).values, n)] * v[ok])
    pm += torch.diag(1.0 - (occ * (v * v)[:, None]).sum(0))
    zz.fill_diagonal_(0.25)
    p = torch.tensor(pairs, device=DEV)
    return {"e": ev[:1].reshape(1, 1), "v": None,
            "corr": {"szsz": zz[p[:, 0], p[:, 1]].cpu().numpy(),
                     "spsm": pm[p[:, 0], p[:, 1]].cpu().numpy().astype(np.complex128),
                     "sz": (sz * (v * v)[:, None]).sum(0).cpu().numpy()}}


def exact(case, seed):
    c = dict(case)
    lat, ks, kind = _lattice(c, seed), _momenta(c), case["kind"]
    n, nd = lat.n_sites, c["nd"]
    if kind == "ground":
        return _ground(c, lat, [(i, j) for i in range(n) for j in range(n)]) if math.comb(n, nd) <= 2000 else None
    if kind == "lanczos":
        return None                       # eigenvectors of 10^6 rows
    if c["k"] == "none":
        return _hphi_u1(lat, nd, _vector(c, math.comb(n, nd), seed))
    # orbit minima over every translation: bounded sizes only
    if math.comb(n, nd) * nd > 2.0e7 or math.comb(n, nd) / n * nd * 6 * n > 4e8:
        return None
    if kind == "smq":
        if math.comb(n, nd + 1) / n > 8e5:
            return None
        q, kq = _transfer(c)
        d = int(_Sectors(n, nd, _dims(c), ks).members[0].numel())
        return _smq(c, lat, _vector(c, d, seed), q, ks[0], kq)
    d = sum(int(m.numel()) for m in _Sectors(n, nd, _dims(c), ks).members)
    phi = _vector(c, d, seed)
    if kind == "corr":
        return _corr_k(c, lat, ks[0], phi, [(0, j) for j in range(n)], _grid_q(c))
    out, dims = _hphi_k(c, lat, ks, phi)
    return {"dims": dims, "psi": out} if kind == "setup" else out
