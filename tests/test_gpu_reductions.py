"""GPU tests of the reductions' inner forms: complex128 sums of squares as 64-bit integers (over
the exponents where they apply, at their limits and beyond) and the sampled top-K selection
(states that the sample fits and states that mislead it)."""
import math

import numpy as np
import pytest

import oracle
from paper_2409_14697_gb300 import inputs
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs():
    require_gpu()
    from paper_2409_14697_gb300 import qs as q
    q.load()
    return q


def _readings(qs, psi):
    n = int(math.log2(psi.size))
    h = qs.qs_create(n, qs.QS_C128)
    try:
        qs.qs_set_amplitudes(h, psi)
        return qs.qs_norm(h), *qs.qs_expectation_z(h)
    finally:
        qs.qs_destroy(h)


# Squares as integers fall short by at most 6 units of 2^-58 of the group's largest square,
# 32 of them in a group; the FP64 sums above add less than 2^-53 per level of 16 or so levels.
REL = 32 * 6 * 2.0 ** -58 + 20 * 2.0 ** -53


@pytest.mark.parametrize("n", [4, 8, 9, 12, 13, 16])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -460, 2.0 ** -464, 2.0 ** 470, 2.0 ** 480, 2.0 ** -511])
def test_integer_sums_of_squares(qs, n, scale):
    """Norm and <Z_q> against exactly rounded host sums: exponents inside the integer form's
    range, on both sides of its limits (biased 560 and 1500) and far outside; spread exponents,
    exact zeros and subnormals in one group."""
    r = np.random.default_rng(n)
    for kind in range(3):
        x = r.standard_normal((1 << n, 2))
        if kind == 1:
            x *= 2.0 ** r.integers(-60, 1, size=x.shape)
        if kind == 2:
            x[r.random(x.shape) < 0.7] = 0.0
            x[r.random(x.shape) < 0.1] = 5e-324 / scale if scale >= 1 else 0.0
        x *= scale
        # powers of two scale squares exactly: sums in units where nothing underflows
        unit = x / scale
        p = [float(a) * float(a) for a in unit.reshape(-1)]
        fine = np.float64(scale) * np.float64(scale)
        norm, ez, nrm = _readings(qs, np.ascontiguousarray(x).view(np.complex128).reshape(-1))
        assert norm == nrm
        if not (2.0 ** -1000 < fine < 2.0 ** 1000):
            assert norm <= 2.0 ** -1000 or scale > 1  # squares near the end of the range
            continue
        want = math.fsum(p)
        assert abs(norm / fine - want) <= REL * want
        prob = np.array(p).reshape(-1, 2).sum(1)
        for q in range(n):
            sign = 1.0 - 2.0 * ((np.arange(1 << n) >> q) & 1)
            assert abs(ez[q] / fine - math.fsum(prob * sign)) <= 3 * REL * want


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_sums_of_non_finite_amplitudes(qs, bad):
    psi = np.ones(1 << 10, dtype=np.complex128)
    psi[77] = bad
    norm, ez, _ = _readings(qs, psi)
    assert not np.isfinite(norm) and not np.any(np.isfinite(ez))


@pytest.mark.parametrize("dtype,n", [(2, 22), (1, 23), (2, 23)])
@pytest.mark.parametrize("k", [1, 300, 2048, 2049, 4096])
def test_top_k_sampled(qs, dtype, n, k):
    """States of 64 MiB and more, whose threshold is sampled: Gaussian, the largest amplitudes in
    one run of indices, every amplitude but a few equal, and large amplitudes on one index in
    64 lines; indices and amplitudes exactly the oracle's."""
    base = inputs.gaussian_state(n, seed=n + k)
    r = np.random.default_rng(k)
    states = [base.copy()]
    run = base.copy()
    run[5000:5000 + 9000] *= 50.0
    states.append(run)
    flat = np.full(1 << n, 2.0 ** -12 + 0j)
    flat[r.integers(0, 1 << n, size=40)] = 2.0 ** -11
    states.append(flat)
    comb = base.copy()
    comb[3::512] *= 30.0
    states.append(comb)
    h = qs.qs_create(n, dtype)
    try:
        for psi in states:
            psi = psi.astype(np.complex128 if dtype == 2 else np.complex64)
            qs.qs_set_amplitudes(h, psi)
            idx, amp = qs.qs_top_amplitudes(h, k)
            widx, wamp = oracle.top_k(psi.astype(np.complex128), n, k)
            assert np.array_equal(idx, widx)
            assert np.array_equal(amp, wamp)
    finally:
        qs.qs_destroy(h)
