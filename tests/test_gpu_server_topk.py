"""GPU test of the top-K that requests of the server run, whose selections follow one another without
a host wait, on states of 64 MiB (the threshold is sampled): indices and amplitudes exactly the
oracle's where the sample fits and where it misleads, with one slot's scratch used over and over."""
import numpy as np
import pytest

import oracle
from paper_2409_14697_gb300 import inputs
from tests.gpu_util import require_gpu
from tests.test_gpu_server import wait

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs():
    require_gpu()
    from paper_2409_14697_gb300 import qs as q
    q.load()
    return q


def _states(n, seed):
    """Gaussian; the largest amplitudes in one run of indices; all but a few equal; all equal; large
    ones on one index in 64 lines."""
    base = inputs.gaussian_state(n, seed=seed)
    r = np.random.default_rng(seed)
    run, comb = base.copy(), base.copy()
    run[5000:5000 + 9000] *= 50.0
    comb[3::512] *= 30.0
    flat = np.full(1 << n, 2.0 ** -12 + 0j)
    few = flat.copy()
    few[r.integers(0, 1 << n, size=40)] = 2.0 ** -11
    return [base, run, few, base[::-1].copy(), flat, comb, base]


@pytest.mark.parametrize("dtype,n", [(2, 22), (1, 23)])
@pytest.mark.parametrize("k", [1, 1024, 4096])
def test_top_k_of_requests(qs, dtype, n, k):
    psis = [p.astype(np.complex128 if dtype == 2 else np.complex64) for p in _states(n, n + k)]
    sv = qs.qs_server_create(2 << 30, max_slots=1)
    try:
        got = [wait(qs, sv, qs.qs_submit(sv, n, dtype, [], top_k=k, init=p), n, k) for p in psis]
    finally:
        qs.qs_server_drain(sv)
        qs.qs_server_destroy(sv)
    for p, r in zip(psis, got):
        idx, amp = oracle.top_k(p.astype(np.complex128), n, k)
        assert np.array_equal(r["top_idx"], idx)
        assert np.array_equal(r["top_amp"], amp)
