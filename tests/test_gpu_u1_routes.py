"""Products without momenta at the edges of the rules that pick their kernel:
segments of fixed upper spins in fp32 (N_down = 3; chains from 483 sites, rings
from 700, up to four neighbours from 512 where bonds are at most N / 24 long),
the row kernel around them, and complex128 with few real entries or N_down = 4.

fp32 against the binary64 product of the same vector: a row adds at most K =
N_down deg + 6 terms, each coefficient and product rounded once: (K + 4) 2^-24 of
the row weight times the largest element.  complex128 against two real products:
(K + 4) 2^-52 of the same.
"""
from __future__ import annotations

import numpy as np
import pytest

import qs3_inputs as qi
from tests.gpu_common import lib_basis, torch_cuda

pytestmark = pytest.mark.gpu


def _weight(spec, nd):
    deg = int(np.bincount(np.concatenate([spec.bi, spec.bj])).max())
    j = max(np.abs(spec.jxy).max(), np.abs(spec.jz).max())
    h = 0.0 if spec.h is None else np.abs(spec.h)
    return deg, np.abs(spec.jz).sum() / 4 + np.sum(h) / 2 + nd * (2 * deg * j + np.max(h))


FP32 = {"chain482": qi.chain(482, periodic=False), "chain483": qi.chain(483, periodic=False), "ring483": qi.chain(483),
        "ring699": qi.chain(699), "ring700": qi.chain(700), "open23": qi.disordered_open_square(23),
        "open24": qi.disordered_open_square(24), "open8x64": qi.hypercubic((8, 64), False, 1.0, 0.7),
        "open2x256": qi.hypercubic((2, 256), False, 1.0, 0.7), "torus24": qi.hypercubic((24, 24), True, 1.0, 0.7)}


@pytest.mark.parametrize("name", FP32)
def test_fp32_segments_and_rows(name):
    torch = torch_cuda()
    spec = FP32[name]
    spec.L = (0, 0, 0)
    b = lib_basis(spec, 3)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(b.total_dim, generator=g, device="cuda", dtype=torch.float32)
    want = b.hphi(x.double())
    deg, w = _weight(spec, 3)
    assert float((b.hphi(x).double() - want).abs().max()) <= (3 * deg + 10) * 2.0 ** -24 * w * float(x.abs().max())


@pytest.mark.parametrize("spec,nd", [(qi.hypercubic((2, 40), False, 1.0, 0.7), 3), (qi.honeycomb(5), 3),
                                     (qi.disordered_open_square(7), 3), (qi.disordered_open_square(6), 4),
                                     (qi.hypercubic((4, 4, 4), False, 1.0, 0.7), 3), (qi.chain(30), 2), (qi.chain(30), 1)],
                         ids=["2x40", "honeycomb5", "open7", "open6_4", "cube4", "ring30_2", "ring30_1"])
def test_complex128_is_two_real_products(spec, nd):
    torch = torch_cuda()
    spec.L, spec.n_sub = (0, 0, 0), 1
    b = lib_basis(spec, nd)
    g = torch.Generator(device="cuda").manual_seed(6)
    x = torch.randn(2, b.total_dim, generator=g, device="cuda", dtype=torch.float64)
    got = b.hphi(torch.complex(x[0], x[1]))
    deg, w = _weight(spec, nd)
    tol = (nd * deg + 10) * 2.0 ** -52 * w * float(x.abs().max())
    assert float((got.real - b.hphi(x[0].contiguous())).abs().max()) <= tol
    assert float((got.imag - b.hphi(x[1].contiguous())).abs().max()) <= tol
