"""GPU test of the complex128 sums of squares at their worst: one group of a thread (the 16 amplitudes
256 apart of a 12-qubit state) with one large real and 31 that lose most of a unit each."""
import math
from fractions import Fraction

import numpy as np
import pytest

from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu

# 32 squares, each short by less than 1.125 units of 2^-56 of the largest or over by at most a quarter;
# the group's conversion and nothing else rounds (all other amplitudes are 0)
BOUND = 32 * 1.125 * 2.0 ** -56 + 2.0 ** -53


def _units_lost(x):
    """Of a real below 1 beside 1.0: what dropping the product's low 64 bits loses, in units."""
    X = int(Fraction(x) * 2 ** 60)
    return float(Fraction(x) ** 2 * 2 ** 56 - (X * X >> 64))


def _smalls():
    """Reals beside 1.0: the low word of X = x 2^60 near 2^32 for small and large high words, with
    bits below X that the shift drops."""
    out = [(2.0 ** h + 2.0 ** 32 - 1.0) * 2.0 ** -60 for h in (40, 42, 45, 50)]
    r = np.random.default_rng(3)
    worst = sorted(r.uniform(2.0 ** -12, 1.0, 20000), key=_units_lost)
    return out + worst[-3:] + [0.9999999 * 2.0 ** -29, math.pi / 4]


@pytest.fixture(scope="module")
def qs():
    require_gpu()
    from paper_2409_14697_gb300 import qs as q
    q.load()
    return q


@pytest.mark.parametrize("thread", [0, 37, 255])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -400, 2.0 ** 400])
def test_one_large_real_beside_many(qs, thread, scale):
    n = 12
    h = qs.qs_create(n, qs.QS_C128)
    try:
        for x in _smalls():
            reals = np.full(32, x)
            reals[2 * (thread % 16)] = 1.0
            psi = np.zeros(1 << n, dtype=np.complex128)
            psi[thread::256] = reals.view(np.complex128) * scale
            qs.qs_set_amplitudes(h, psi)
            norm = qs.qs_norm(h)
            ez, nrm = qs.qs_expectation_z(h)
            want = 1 + 31 * Fraction(x) ** 2
            got = Fraction(norm) / Fraction(scale) ** 2
            assert norm == nrm
            assert abs(float(got - want)) <= BOUND * float(want), x
            for q in range(n):  # masses of the high bits come from the same sums, <Z> is total - 2 mass
                bits = (np.arange(1 << n)[thread::256] >> q) & 1
                sign = 1 - 2 * bits.astype(int)
                exact = sum(int(sign[j // 2]) * Fraction(float(reals[j])) ** 2 for j in range(32))
                got = Fraction(float(ez[q])) / Fraction(scale) ** 2
                assert abs(float(got - exact)) <= 4 * BOUND * float(want), (x, q)
    finally:
        qs.qs_destroy(h)
