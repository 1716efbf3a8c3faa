"""GPU tests of the corrections of FP32 rounding in complex64 register phases: states that a
circuit's roundings leave alone stay as they are (alone and in a batch), and the norm of a state
after many equal rotations."""
import numpy as np
import pytest

from paper_2409_14697_gb300 import inputs
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu

CAP = 6e-6   # largest correction of a call for roundings that depend on the state's populations
ULP = 6e-8   # 2^-24


@pytest.fixture(scope="module")
def qs():
    require_gpu()
    from paper_2409_14697_gb300 import qs as q
    q.load()
    return q


def _phases_on_zeros(n, theta):
    """3600 phases of one angle on qubits in |0>: the amplitude of |0...0> stays 1."""
    gates = [("rx", (n - 1,), (0.0,))]
    for i in range(1800):
        gates.append(("cp", (i % (n - 1), (i + 1) % (n - 1)), (theta,)))
        gates.append(("p", (i % (n - 1),), (theta,)))
    return gates


@pytest.mark.parametrize("theta", [0.8043, 1.0])
def test_phases_on_zeros_keep_the_state(qs, theta):
    circuits = [(n, _phases_on_zeros(n, theta)) for n in (10, 11, 12)]
    got = []
    for n, gates in circuits:
        h = qs.qs_create(n, qs.QS_C64)
        try:
            qs.qs_apply_circuit(h, gates)
            got.append(qs.qs_amplitudes(h))
        finally:
            qs.qs_destroy(h)
    b = qs.qs_batch_create(circuits, qs.QS_C64)
    try:
        qs.qs_batch_run(b)
        qs.qs_batch_synchronize(b)
        got += [qs.qs_batch_amplitudes(b, i, n) for i, (n, _) in enumerate(circuits)]
    finally:
        qs.qs_batch_destroy(b)
    for psi in got:
        assert abs(psi[0] - 1.0) <= CAP + 2 * ULP   # the factor and its own rounding
        assert np.count_nonzero(psi[1:]) == 0


def test_equal_rotations_keep_the_norm_of_large_states(qs):
    """16 Trotter steps at 22 qubits, phases in layers.  What the FP32 reals of the matrices do to the
    norm is divided out up to the cap; each step's tables may leave a rounding of their own."""
    n, steps, dt, field = 22, 16, 0.05, 1.0
    half = dt * field   # RX by twice that
    c, s = np.float32(np.cos(half)), np.float32(np.sin(half))
    total = 0.5 * (float(c) ** 2 + float(s) ** 2 - 1.0) * n * steps
    h = qs.qs_create(n, qs.QS_C64)
    try:
        qs.qs_apply_circuit(h, inputs.tfim(n, steps, dt=dt, h=field))
        norm = qs.qs_norm(h)
    finally:
        qs.qs_destroy(h)
    assert abs(norm - 1.0) <= 2 * max(0.0, abs(total) - CAP) + 2 * 2 * steps * ULP
