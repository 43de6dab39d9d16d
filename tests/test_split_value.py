"""The recombination of a tile's digit sums (split_value) against exact
integers: operands whose digits add up in step (constants, all-ones
mantissas) over 16 to 256 real terms, either sign.  The value is the sum in
units of 2^58 (2^59 above 128 terms) digit units, its lowest part rounded to
that unit, then rounded to a double: within half a unit and half an ulp."""
import ctypes
from fractions import Fraction

import numpy as np
import pytest

from tests import split_device


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return split_device.load(tmp_path_factory.mktemp("split"))


def digits(n):
    """Seven digits of n < 2^57 in base 256, the lower six in -128 .. 127."""
    out = []
    for _ in range(6):
        d = (n + 128) % 256 - 128
        out.append(d)
        n = (n - d) // 256
    return [n] + out[::-1]


def mantissas():
    rng = np.random.default_rng(5)
    full = (1 << 53) - 1
    return [full, 1 << 52, full - 127, 0x1FF7F7F7F7F7F8, 0x1F8080808080 << 5] + \
        [int(v) for v in rng.integers(1 << 52, 1 << 53, size=40)]


@pytest.mark.parametrize("ks", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("sign", [1, -1])
def test_constant_operands(lib, ks, sign):
    terms, unit = 16 * ks, 1 << (59 if ks > 8 else 58)
    ms = mantissas()
    for a, b in list(zip(ms, ms)) + list(zip(ms, ms[1:])):
        da, db = digits(a << 4), digits(b << 4)
        sums = [sign * terms * sum(da[i] * db[d - i] for i in range(d + 1)) for d in range(7)]
        exact = Fraction(sum(s << (8 * (12 - d)) for d, s in enumerate(sums)), unit)
        got = Fraction(lib.split_value_host(ks, (ctypes.c_int * 7)(*sums)))
        assert abs(got - exact) <= Fraction(1, 2) + abs(exact) / (1 << 53), (hex(a), hex(b))
