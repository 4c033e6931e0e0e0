"""The rows of a momentum sector are counted before anything is allocated: a
sector of 2^32 rows or more is refused with OVERFLOW for every momentum, and
the number in the message is the character sum written out translation by
translation.  Smaller ones go on to allocate (an injected failure shows it),
so none of this needs a GPU."""
from __future__ import annotations

import cmath
import math
import re

import pytest

import qs3_inputs as qi

OVERFLOW, OOM = -2, -4


def _rows(dims, nd, k):
    n = math.prod(dims)
    total = 0
    for t in ((x, y, z) for z in range(dims[2]) for y in range(dims[1]) for x in range(dims[0])):
        o = math.lcm(*(l // math.gcd(l, v) for l, v in zip(dims, t)))
        fixed = math.comb(n // o, nd // o) if nd % o == 0 else 0
        phase = sum(a * b * (n // l) for a, b, l in zip(k, t, dims)) % n
        total += fixed if phase == 0 else fixed * cmath.exp(2j * math.pi * phase / n).real
    return round(total / n)


def _create(dims, nd, ks):
    import paper_2107_00872_gb300 as qs3
    prev = qs3.inject_alloc_failure(0)
    try:
        with pytest.raises(qs3.QS3Error) as e:
            qs3.Basis(qi.hypercubic(dims, True), nd, ks)
        return e.value.status, qs3.load().qs3_last_error().decode()
    finally:
        qs3.inject_alloc_failure(prev)


@pytest.mark.parametrize("dims,nd,ks", [
    ((12, 12, 6), 5, [(1, 0, 0)]), ((12, 12, 6), 5, [(0, 0, 0)]), ((7, 7, 7), 6, [(1, 0, 0)]),
    ((34, 25, 1), 5, [(0, 0, 0), (17, 5, 0)]), ((50, 17, 1), 5, [(3, 2, 0)]), ((53, 6, 1), 6, [(1, 3, 0)])])
def test_sector_beyond_32_bit_rows(dims, nd, ks):
    st, msg = _create(dims, nd, ks)
    assert st == OVERFLOW
    n = _rows(dims, nd, ks[0])
    assert n >= 2 ** 32 and int(re.search(r"dimension (\d+)", msg).group(1)) == n


@pytest.mark.parametrize("dims,nd,k", [((33, 25, 1), 5, (1, 0, 0)), ((12, 12, 5), 5, (1, 0, 0)), ((7, 7, 6), 6, (0, 0, 3))])
def test_sector_within_32_bit_rows(dims, nd, k):
    assert 2 ** 30 < _rows(dims, nd, k) < 2 ** 32
    assert _create(dims, nd, [k])[0] == OOM
