"""The kernels that a rule on sizes picks, at the edges of their ranges: each
is compared with the general path or the oracle on inputs where it can go
wrong (tile and chunk remainders, degrees, periodic wraps, stabilisers, both
key widths, coordinate ranges)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle as orc
import qs3_inputs as qi
from tests.gpu_common import gaussian, lib_basis, olat, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _row_weight(spec, nd):
    """A bound of sum_j |H_ij| over all rows: the diagonal's constant and site
    terms, and N_down sites' hops and J^z."""
    deg = np.bincount(np.concatenate([spec.bi, spec.bj]), minlength=spec.n_sites).max()
    j = max(np.abs(spec.jxy).max(), np.abs(spec.jz).max())
    h = 0.0 if spec.h is None else np.abs(spec.h)
    return np.abs(spec.jz).sum() / 4 + np.sum(h) / 2 + nd * (2 * deg * j + np.max(h))


# fp32 rows in segments of fixed upper spins (N_down = 3, mean segment from 160
# rows): against the binary64 product of the same vector.  A row adds at most K
# = 3 deg + 6 terms, each coefficient and product rounded once: (K + 4) 2^-24 of
# the row weight times the largest element.
@pytest.mark.parametrize("spec", [qi.disordered_open_square(22), qi.chain(483), qi.chain(484, periodic=False),
                                  qi.hypercubic((8, 8, 8), False, 1.0, 0.7), qi.hypercubic((22, 22), True, 1.0, 0.7)],
                         ids=["open22", "ring483", "chain484", "cube8", "torus22"])
@pytest.mark.parametrize("cplx", [False, True])
def test_segments_fp32(spec, cplx):
    torch = torch_cuda()
    spec.L = (0, 0, 0)
    b = lib_basis(spec, 3)
    d = b.total_dim
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(d * (2 if cplx else 1), generator=g, device="cuda", dtype=torch.float32)
    y = torch.view_as_complex(x.view(d, 2)) if cplx else x
    got = b.hphi(y)
    want = b.hphi(y.to(torch.complex128 if cplx else torch.float64))
    deg = np.bincount(np.concatenate([spec.bi, spec.bj])).max()
    tol = (3 * deg + 10) * 2.0 ** -24 * _row_weight(spec, 3) * float(x.abs().max()) * (2 if cplx else 1)
    assert float((got.to(want.dtype) - want).abs().max()) <= tol


# sectors taken from one enumeration: ranks and stabilisers of every momentum
@pytest.mark.parametrize("spec,nd", [(qi.chain(12), 1), (qi.chain(12), 4), (qi.square(4, 3), 3), (qi.square(4), 4),
                                     (qi.hypercubic((3, 2, 4), True), 4), (qi.honeycomb(3), 3), (qi.kagome(2, 3), 4)],
                         ids=["ring12_1", "ring12_4", "4x3", "4x4", "3x2x4", "honeycomb3", "kagome2x3"])
def test_all_sectors_at_once(spec, nd):
    torch_cuda()
    ks = qi.all_k(spec.L)
    b = lib_basis(spec, nd, ks)
    for s, k in enumerate(ks):
        sec = orc.mk_list(olat(spec), nd, k)
        r, st = b.ranks(s)
        np.testing.assert_array_equal(r, sec.rank0)
        np.testing.assert_array_equal(st, sec.stab)


# the representative search on occupation masks (up to 32 cells along an axis)
# and without them, through the bucket index, against the table
@pytest.mark.parametrize("dims,nd", [((32,), 4), ((33,), 4), ((32, 2), 3), ((2, 33), 3), ((5, 4, 3), 5)])
def test_search_equals_table(dims, nd):
    torch = torch_cuda()
    spec = qi.hypercubic(dims, True, 1.0, 0.8)
    ks = [(0, 0, 0), (1, 0, 0), (dims[0] // 2, 0, 0)]
    b = lib_basis(spec, nd, ks)
    phi = to_dev(gaussian(3, b.total_dim, True), torch.complex128)
    assert b.rep_table()
    ref = b.hphi(phi)
    assert not b.rep_table(0)
    assert torch.equal(b.hphi(phi), ref)


# origin forms (no table: 2^20 orbits or more), 32- and 64-bit keys, against the
# terms that the representative search enumerates: the same bits
@pytest.mark.parametrize("dims,nd,ks", [((64,), 6, [(3, 0, 0), (0, 0, 0)]), ((13, 5), 6, [(6, 2, 0)]),
                                        ((300,), 4, [(150, 0, 0)]), ((5, 5, 5), 5, [(0, 0, 0), (2, 1, 4)])])
def test_origin_forms_equal_search(dims, nd, ks):
    torch = torch_cuda()
    b = lib_basis(qi.hypercubic(dims, True, 1.0, 0.9), nd, ks)
    assert not b.rep_table()
    g = torch.Generator(device="cuda").manual_seed(9)
    phi = torch.view_as_complex(torch.randn(b.total_dim, 2, generator=g, device="cuda", dtype=torch.float64))
    ref = b.hphi(phi)
    assert b.store_terms(1) > 0
    assert torch.equal(b.hphi(phi), ref)


# the orbit-batched products against one sector at a time
@pytest.mark.parametrize("spec,nd", [(qi.square(5, 4), 4), (qi.square(6), 3), (qi.hypercubic((3, 3, 4), True), 2),
                                     (qi.triangular(4, 6), 3)], ids=["5x4", "6x6", "3x3x4", "tri4x6"])
@pytest.mark.parametrize("nk", [2, 9, 0])
def test_batched_sectors_equal_single(spec, nd, nk):
    torch = torch_cuda()
    ks = qi.all_k(spec.L)
    ks = ks[: nk or len(ks)]
    b = lib_basis(spec, nd, ks)
    for dt in (torch.complex128, torch.complex64):
        phi = to_dev(gaussian(4, b.total_dim, True), dt)
        got = b.hphi(phi)
        for s, k in enumerate(ks):
            one = lib_basis(spec, nd, [k])
            lo, hi = b.offsets[s], b.offsets[s + 1]
            x = phi[lo:hi].contiguous()
            assert torch.equal(one.hphi(x), got[lo:hi])
            one.rep_table(0)                            # the row kernel with the search
            assert torch.equal(one.hphi(x), got[lo:hi])


# two-point functions and S^-_q, S^+_q by the table and by the search.  Each is a
# sum of at most N (N - 1) binary64 terms of unit weight on a unit vector.
@pytest.mark.parametrize("dims,nd,k", [((4, 3), 3, (1, 2, 0)), ((5, 5), 4, (0, 0, 0)), ((9,), 2, (4, 0, 0)),
                                       ((3, 2, 4), 4, (0, 1, 2))])
def test_observables_table_and_search(dims, nd, k):
    torch = torch_cuda()
    import paper_2107_00872_gb300 as qs3
    spec = qi.hypercubic(dims, True)
    n = spec.n_sites
    q = (1, 0, 0)
    kq = tuple((k[a] + q[a]) % spec.L[a] for a in range(3))
    b, up = lib_basis(spec, nd, [k]), lib_basis(spec, nd + 1, [kq])
    v = gaussian(7, b.total_dim, True)
    phi = to_dev(v / np.linalg.norm(v), torch.complex128)
    u = gaussian(8, up.total_dim, True)
    top = to_dev(u / np.linalg.norm(u), torch.complex128)
    back = tuple((-x) % spec.L[a] for a, x in enumerate(q))
    pairs, qs = [(0, j) for j in range(n)], np.array([[0.3, 0.1, 0.2], [2 * np.pi / dims[0], 0, 0]])

    def all_of():
        c = b.correlations(phi, 0, pairs=pairs, q=qs, local=True)
        return [*c.values(), qs3.smq(b, 0, phi, up, 0, q).cpu().numpy(),
                qs3.sq_apply(qs3.OP_SPLUS, up, 0, top, b, 0, back).cpu().numpy()]

    got = all_of()
    b.rep_table(0)
    up.rep_table(0)
    for x, y in zip(got, all_of()):
        assert np.max(np.abs(x - y)) <= n * n * 2.0 ** -52


# Lanczos steps of few chunks: 1, 2, 8 (sums formed in place) and 9 chunks of
# 2048 rows.  The ground state of the ring against its momentum sectors' dense
# spectra; graph replay and direct launches agree bit for bit.
@pytest.mark.parametrize("n", [24, 25, 47, 49])
def test_few_chunk_lanczos(n):
    torch_cuda()
    import paper_2107_00872_gb300 as qs3
    spec = qi.chain(n)
    ks = lib_basis(spec, 3, qi.all_k(spec.L))
    e0 = min(float(ks.full_diag(s)[0][0]) for s in range(ks.n_sectors) if ks.dims[s])
    b = lib_basis(spec, 3)
    ev = []
    for graphs in (True, False):
        e, _, info = b.lanczos(qs3.SolveOpts(n_max=200, eps=1e-14, res_tol=1e-12, use_graphs=graphs))
        assert info["status"] == "QS3_OK" and info["max_residual"] <= 1e-9 * max(1.0, abs(e0))
        ev.append(float(e[0, 0]))
    assert ev[0] == ev[1]
    assert abs(ev[0] - e0) <= 1e-11 * max(1.0, abs(e0))


def test_integer_product_on_two_streams():
    """Scratch of concurrent calls comes from the pool in stream order."""
    torch = torch_cuda()
    b = lib_basis(qi.square(6), 4, qi.all_k((6, 6, 1)))
    phi = [to_dev(gaussian(s, b.total_dim, True), torch.complex128) for s in (1, 2)]
    ref = [b.hphi(x, integer=True) for x in phi]
    torch.cuda.synchronize()
    st = [torch.cuda.Stream() for _ in phi]
    for _ in range(8):
        out = [torch.empty_like(x) for x in phi]
        torch.cuda.synchronize()
        for x, o, s in zip(phi, out, st):
            b.hphi(x, o, stream=s, integer=True)
        torch.cuda.synchronize()
        assert all(torch.equal(a, r) for a, r in zip(out, ref))
