"""The index over the rows of many sectors, built for a few sectors at a time:
products that look their targets up in it against the representative table,
and a basis with more than 2^31 prefixes."""
from __future__ import annotations

import math

import numpy as np
import pytest

import qs3_inputs as qi
from tests.gpu_common import lib_basis, torch_cuda

pytestmark = pytest.mark.gpu


def _randn(torch, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(d, 2, generator=g, device="cuda", dtype=torch.float32))


# 12x12, N_down = 4, all 144 momenta: about 11.6 million entries, several groups; 9x5
# and 6x4 stay within one (two-site and one-site prefixes, lists and rows)
@pytest.mark.parametrize("dims,nd", [((12, 12), 4), ((9, 5), 4), ((6, 4), 2), ((9, 5), 3), ((3, 2), 2), ((4, 2), 3)])
def test_index_equals_table(dims, nd):
    torch = torch_cuda()
    spec = qi.hypercubic(dims, True, 1.0, 0.8)
    b = lib_basis(spec, nd, qi.all_k(spec.L))
    phi = _randn(torch, b.total_dim, 3)
    assert b.rep_table()
    ref = b.hphi(phi)
    assert not b.rep_table(0)
    assert torch.equal(b.hphi(phi), ref)


def test_index_of_many_prefixes():
    torch = torch_cuda()
    spec = qi.hypercubic((41, 41), True)
    n, ks = spec.n_sites, qi.all_k(spec.L)
    assert n * (n * (n - 1) // 2) > 2 ** 31
    b = lib_basis(spec, 3, ks)
    assert b.total_dim == math.comb(n, 3) and not b.rep_table()
    phi = _randn(torch, b.total_dim, 4)
    psi = b.hphi(phi)
    for s in (0, 1, 1000, n - 1):
        one = lib_basis(spec, 3, [ks[s]])           # found by its origin forms
        lo, hi = b.offsets[s], b.offsets[s + 1]
        np.testing.assert_array_equal(b.ranks(s)[0], one.ranks()[0])
        assert torch.equal(one.hphi(phi[lo:hi].contiguous()), psi[lo:hi])


# a basis of few rows is bound by the allocations of its creation, whose number
# does not depend on the sectors; what the destruction leaves of the scratch is
# mapped no more by the next creation
@pytest.mark.parametrize("nk", [1, 4, 25])
def test_creation_allocates_little(nk):
    torch = torch_cuda()
    import paper_2107_00872_gb300 as qs3
    spec = qi.square(5)

    def create():
        qs3.inject_alloc_failure(1000)
        try:
            b = lib_basis(spec, 3, qi.all_k(spec.L)[:nk])
        finally:
            left = qs3.inject_alloc_failure(-1)
        b.close()
        return 1000 - left

    create()
    free = torch.cuda.mem_get_info()[0]
    assert create() <= 24
    assert abs(torch.cuda.mem_get_info()[0] - free) <= 4 << 20


# a basis without the table holds the origin forms of its rows, about 20 bytes
# each, and gives them back with mode 0; the search finds the same bits
def test_origin_forms_are_given_back():
    torch = torch_cuda()
    b = lib_basis(qi.hypercubic((13, 5), True, 1.0, 0.9), 6, [(6, 2, 0)])
    assert not b.rep_table()
    phi = _randn(torch, b.total_dim, 5)
    ref = [b.hphi(x) for x in (phi, phi.to(torch.complex128))]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    assert not b.rep_table(0)
    assert torch.cuda.mem_get_info()[0] - free >= 16 * b.total_dim
    for x, r in zip((phi, phi.to(torch.complex128)), ref):
        assert torch.equal(b.hphi(x), r)
