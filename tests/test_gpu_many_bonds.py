"""Lattices of many equal bonds (all pairs of a ring or a square): the products
whose rows have hundreds of terms, against the binary64 FMA product.

A row's sum of n terms, each of modulus at most |phi|max J / 2: the FMA product
rounds every partial sum, the integer product each term on the grid of the
largest and each fold once, so they differ by at most n^2 2^-52 of that modulus;
the diagonal adds a few roundings of its own weight, (n + N_down^2 + N^2) |J^z|.
"""
from __future__ import annotations

import numpy as np
import pytest

import qs3_inputs as qi
from tests.gpu_common import lib_basis, torch_cuda

pytestmark = pytest.mark.gpu


def _all_pairs(dims):
    n = int(np.prod(dims))
    bi, bj = np.triu_indices(n, 1)
    L = tuple(dims) + (1,) * (3 - len(dims))
    return qi.LatticeSpec(n, bi.astype(np.int32), bj.astype(np.int32), np.ones(len(bi)), np.full(len(bi), 0.01), None,
                          L, "all pairs")


def _tol(n_sites, nd, phi):
    n = nd * (n_sites - nd)
    return (n * n * 0.5 + 8 * 0.01 * n_sites ** 2) * 2.0 ** -52 * float(phi.abs().max())


# rows of equal elements just below a power of two: every one of the 1028 terms
# is the largest that the grid holds, at k = 0 in step
@pytest.mark.parametrize("n,nd", [(261, 4), (100, 5)])
def test_integer_product_of_many_terms(n, nd):
    torch = torch_cuda()
    b = lib_basis(_all_pairs((n,)), nd, [(0, 0, 0)])
    phi = torch.full((b.total_dim,), (1 - 2.0 ** -53) * (1 - 1j), dtype=torch.complex128, device="cuda")
    assert float((b.hphi(phi, integer=True) - b.hphi(phi)).abs().max()) <= _tol(n, nd, phi)


# hop lists beyond shared memory (192 hops a row) over several sectors: the
# product, and the binary64 solve that uses it, against binary64 FMAs
def test_many_bonds_over_several_sectors():
    torch = torch_cuda()
    import paper_2107_00872_gb300 as qs3
    spec, nd = _all_pairs((7, 7)), 4
    b = lib_basis(spec, nd, [(0, 0, 0), (1, 3, 0)])
    g = torch.Generator(device="cuda").manual_seed(2)
    phi = torch.view_as_complex(torch.randn(b.total_dim, 2, generator=g, device="cuda", dtype=torch.float64))
    got = b.hphi(phi, integer=True)
    assert float((got - b.hphi(phi)).abs().max()) <= _tol(49, nd, phi)
    e = []
    for strict in (False, True):
        ev, _, info = b.lanczos(qs3.SolveOpts(n_max=60, eps=1e-13, res_tol=1e-10, strict64=strict))
        assert info["status"] == "QS3_OK"
        e.append(ev[:, 0])
    assert np.max(np.abs(e[0] - e[1])) <= 1e-11 * np.max(np.abs(e[1]))


# lattices of equal bonds to the nearest `degree` sites, where the number of
# sectors decides between the orbit-batched kernel and the row kernel: all
# momenta at once against one at a time, the same bits
@pytest.mark.parametrize("dims,nd,degree", [((8, 8), 4, 10), ((8, 8), 4, 14), ((8, 8), 4, 20), ((8, 8), 4, 28),
                                            ((5, 5), 6, 8), ((10, 10), 3, 18)])
def test_batched_equals_single_with_many_bonds(dims, nd, degree):
    torch = torch_cuda()
    lx, ly = dims
    near = sorted((min(x, lx - x) ** 2 + min(y, ly - y) ** 2, x, y) for x in range(lx) for y in range(ly))[1:]
    d = set()
    for _, x, y in near:
        if len(d) < degree and (-x % lx, -y % ly) != (x, y):
            d |= {(x, y), (-x % lx, -y % ly)}
    pairs = [(r, (r % lx + x) % lx + lx * ((r // lx + y) % ly)) for r in range(lx * ly) for x, y in sorted(d)]
    b = np.array([p for p in pairs if p[0] < p[1]], np.int32)
    spec = qi.LatticeSpec(lx * ly, b[:, 0].copy(), b[:, 1].copy(), np.full(len(b), 0.7), np.full(len(b), 0.9), None,
                          (lx, ly, 1), "near")
    ks = qi.all_k(spec.L)
    both = lib_basis(spec, nd, ks)
    g = torch.Generator(device="cuda").manual_seed(6)
    x = torch.view_as_complex(torch.randn(both.total_dim, 2, generator=g, device="cuda", dtype=torch.float64))
    for phi in (x, x.to(torch.complex64)):
        psi = both.hphi(phi)
        for s in (0, 1, len(ks) // 2):
            lo, hi = both.offsets[s], both.offsets[s + 1]
            assert torch.equal(lib_basis(spec, nd, [ks[s]]).hphi(phi[lo:hi].contiguous()), psi[lo:hi])
    psi = both.hphi(x, integer=True)
    for s in (0, 1, len(ks) // 2):
        lo, hi = both.offsets[s], both.offsets[s + 1]
        one = lib_basis(spec, nd, [ks[s]]).hphi(x[lo:hi].contiguous(), integer=True)
        assert float((one - psi[lo:hi]).abs().max()) <= 2 * _tol(lx * ly, nd, x)
