"""Momentum-sector products on lattices whose couplings differ from axis to axis,
in a uniform field: the origin forms' per-bond amplitudes and diagonal sums, and
the orbit-batched kernels' diagonal sums, which lattices of one J^xy and one J^z
do not reach.

The reference is the stored terms (origin forms), or one sector at a time through
the representative search (batches).  A row adds at most K = N_down deg terms and
N_down (deg + 1) + 1 diagonal ones, each rounded at most twice: 4 (K + 2) units in
the last place of the row weight times the largest element.
"""
from __future__ import annotations

import numpy as np
import pytest

import qs3_inputs as qi
from tests.gpu_common import lib_basis, torch_cuda

pytestmark = pytest.mark.gpu


def _per_axis(dims, jxy, jz, field):
    """J^xy and J^z by the axis of each bond."""
    spec = qi.hypercubic(dims, True)
    strides = np.cumprod((1,) + tuple(dims))[:-1]
    axis = []
    for i, j in zip(spec.bi, spec.bj):
        ci, cj = [[int(r) // s % d for s, d in zip(strides, dims)] for r in (i, j)]
        axis.append([a for a in range(len(dims)) if ci[a] != cj[a]][0])
    spec.jxy = np.array([jxy[a] for a in axis])
    spec.jz = np.array([jz[a] for a in axis])
    spec.h = np.full(spec.n_sites, field)
    return spec


def _tol(spec, nd, phi):
    deg = int(np.bincount(np.concatenate([spec.bi, spec.bj])).max())
    weight = (np.abs(spec.jz).sum() / 4 + np.abs(spec.h).sum() / 2
              + nd * (2 * deg * max(np.abs(spec.jxy).max(), np.abs(spec.jz).max()) + np.abs(spec.h).max()))
    eps = 2.0 ** -24 if "64" in str(phi.dtype) else 2.0 ** -53
    return 4 * (nd * deg + 2) * eps * weight * float(phi.abs().max())


def _randn(torch, d, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(d, 2, generator=g, device="cuda", dtype=torch.float64))


@pytest.mark.parametrize("dims,nd,ks", [((13, 5), 6, [(6, 2, 0)]), ((5, 5, 5), 5, [(0, 0, 0), (2, 1, 4)])])
@pytest.mark.parametrize("jxy", [(1.0, 0.7, 1.3), (1.0, 1.0, 1.0)], ids=["bond amplitudes", "one amplitude"])
def test_origin_forms(dims, nd, ks, jxy):
    torch = torch_cuda()
    spec = _per_axis(dims, jxy, (0.9, 0.4, 1.1), 0.3)
    b = lib_basis(spec, nd, ks)
    assert not b.rep_table()
    x = _randn(torch, b.total_dim, 9)
    got = [b.hphi(phi) for phi in (x, x.to(torch.complex64))]
    assert b.store_terms(1) > 0
    ref = b.hphi(x)
    for phi, psi in zip((x, x.to(torch.complex64)), got):
        assert float((psi - ref).abs().max()) <= _tol(spec, nd, phi)


@pytest.mark.parametrize("dims,nd", [((6, 6), 3), ((5, 4), 4), ((3, 3, 4), 2)])
def test_batched_sectors(dims, nd):
    torch = torch_cuda()
    spec = _per_axis(dims, (0.8, 0.8, 0.8), (0.9, 0.4, 1.1), 0.3)
    ks = qi.all_k(spec.L)
    b = lib_basis(spec, nd, ks)
    x = _randn(torch, b.total_dim, 4)
    ref = []
    for s, k in enumerate(ks):
        one = lib_basis(spec, nd, [k])
        one.rep_table(0)
        ref.append(one.hphi(x[b.offsets[s]:b.offsets[s + 1]].contiguous()))
    ref = torch.cat(ref)
    assert torch.equal(b.hphi(x), ref)
    for phi, integer in ((x.to(torch.complex64), False), (x, True)):
        assert float((b.hphi(phi, integer=integer) - ref).abs().max()) <= _tol(spec, nd, phi)
