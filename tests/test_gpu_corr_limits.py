"""Correlations near the largest lattices: what the kernel needs of shared memory
(the block's sums, binomial rows and coordinates) is what the call is checked
against.  N_down = 1 has a closed form, the one-spin state of momentum K: <s^+_0
s^-_d> = e^{i K d} / N up to orientation, <s^z s^z> = 1/4 - 1/N; N_down = 2 a sum
rule.
"""
from __future__ import annotations

import numpy as np
import pytest

import qs3_inputs as qi
from tests.gpu_common import lib_basis, torch_cuda

pytestmark = pytest.mark.gpu


def test_one_spin():
    torch = torch_cuda()
    lx, n, k = 1950, 3900, 5
    b = lib_basis(qi.hypercubic((lx, 2), True), 1, [(k, 0, 0)])
    assert b.total_dim == 1
    phi = torch.ones(1, dtype=torch.complex128, device="cuda")
    pairs = [(0, d) for d in (1, 7, 1950, 3899)]
    c = b.correlations(phi, 0, pairs=pairs)
    want = np.array([2 * np.pi * ((k * (d % lx)) % lx) / lx for _, d in pairs])
    assert np.max(np.abs(np.asarray(c["szsz"]) - (0.25 - 1 / n))) <= 1e-15
    assert np.max(np.abs(c["spsm"].real - np.cos(want) / n)) <= 1e-15
    assert np.max(np.abs(np.abs(c["spsm"].imag) - np.abs(np.sin(want)) / n)) <= 1e-15


def test_two_spins():
    torch = torch_cuda()
    n = 3400
    b = lib_basis(qi.hypercubic((1700, 2), True), 2, [(0, 0, 0)])
    g = torch.Generator(device="cuda").manual_seed(1)
    phi = torch.view_as_complex(torch.randn(b.total_dim, 2, generator=g, device="cuda", dtype=torch.float64))
    c = b.correlations(phi, 0, pairs=[(0, j) for j in range(1, n)])
    # sum_j <s^z_0 s^z_j> = <s^z_0> S^z - 1/4 over j != 0, with <s^z_0> = 1/2 - 2/N, S^z = N/2 - 2
    assert abs(float(np.sum(c["szsz"])) - ((0.5 - 2 / n) * (n / 2 - 2) - 0.25)) <= 1e-11 * n
