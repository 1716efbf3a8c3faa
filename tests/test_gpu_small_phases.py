"""GPU parity of complex64 states of 10 to 12 qubits, which run their register phases on the
first 32 to 128 threads of a block (9 and 13 beside them), alone and in a batch, against the
oracle: every gate type a phase holds and the ones it leaves to sweeps, and equal angles repeated,
whose FP32 rounding the last member of a pass takes back."""
import numpy as np
import pytest

import oracle
from paper_2409_14697_gb300 import inputs
from tests.gpu_util import TOL_C64, fidelity_gap, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qs():
    require_gpu()
    from paper_2409_14697_gb300 import qs as q
    q.load()
    return q


def _gates(n):
    gates = inputs.random_circuit(n, 150, seed=n) + inputs.brickwork(n, 5, seed=n) + inputs.qft(n)
    gates.append(("dense", (2, n - 1), inputs.random_unitary(2, seed=n)))
    return gates + inputs.qaoa_complete(n, 2, seed=n) + inputs.random_circuit(n, 60, seed=3 * n)


@pytest.mark.parametrize("n", [9, 10, 11, 12, 13])
@pytest.mark.parametrize("fuse_k", [0, 2])
def test_one_tile_states(qs, n, fuse_k):
    gates = _gates(n)
    psi0 = inputs.gaussian_state(n, seed=n).astype(np.complex64)
    want = oracle.run(psi0.astype(np.complex128), n, gates)
    h = qs.qs_create(n, qs.QS_C64)
    try:
        qs.qs_set_amplitudes(h, psi0)
        qs.qs_apply_circuit(h, gates, qs.options(fuse_k=fuse_k))
        got = qs.qs_amplitudes(h)
    finally:
        qs.qs_destroy(h)
    assert np.max(np.abs(got - want)) <= TOL_C64
    assert fidelity_gap(got, want) <= 1e-6


def test_one_tile_states_in_a_batch(qs):
    circuits = [(n, _gates(n)) for n in (9, 10, 11, 12, 13, 14)] + [(12, inputs.tfim(12, 20))]
    b = qs.qs_batch_create(circuits, qs.QS_C64)
    try:
        for _ in range(2):
            qs.qs_batch_run(b)
            qs.qs_batch_synchronize(b)
            for i, (n, gates) in enumerate(circuits):
                want = oracle.run(oracle.zero_state(n), n, gates)
                assert np.max(np.abs(qs.qs_batch_amplitudes(b, i, n) - want)) <= TOL_C64
    finally:
        qs.qs_batch_destroy(b)


@pytest.mark.parametrize("n", [10, 12])
def test_repeated_angles_keep_the_norm(qs, n):
    """200 Trotter steps of equal angles: FP32-rounded matrices would change the norm by up to
    2 * 200 * 6e-8 n = 2.4e-5 n; the correction leaves single roundings, sqrt(400 n) 6e-8 or so."""
    gates = inputs.tfim(n, 200, dt=0.05)
    h = qs.qs_create(n, qs.QS_C64)
    try:
        qs.qs_apply_circuit(h, gates)
        norm = qs.qs_norm(h)
    finally:
        qs.qs_destroy(h)
    assert abs(norm - 1.0) <= 10 * np.sqrt(400 * n) * 6e-8
