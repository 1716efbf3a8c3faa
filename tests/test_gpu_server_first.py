"""GPU test of a process's first requests: small requests submitted with a large one, in a process
that has launched nothing before, do not wait for it."""
import json
import os
import subprocess
import sys
from pathlib import Path

import pytest

from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu

SCRIPT = """
import json, time
from paper_2409_14697_gb300 import inputs, qs
n_big = 26
sv = qs.qs_server_create(8 << 30, max_slots=2, small_slots=4, small_max_qubits=16)
big = qs.gate_records(inputs.brickwork(n_big, 60, seed=1))
smalls = [(n, qs.gate_records(inputs.brickwork(n, 8, seed=n))) for n in (10, 12, 14, 16)]
t_big = qs.qs_submit(sv, n_big, qs.QS_C128, big, top_k=64)
t_small = [qs.qs_submit(sv, n, dt, g, top_k=64) for dt in (qs.QS_C64, qs.QS_C128) for n, g in smalls]
def wait(t, n):
    while True:
        r = qs.qs_poll(sv, t, n, 64)
        if r is not None:
            return r["latency_s"]
        time.sleep(2e-4)
small = [wait(t, smalls[i % 4][0]) for i, t in enumerate(t_small)]
print(json.dumps({"small": small, "big": wait(t_big, n_big)}))
qs.qs_server_drain(sv)
qs.qs_server_destroy(sv)
"""


def test_first_requests_of_a_process_overlap():
    require_gpu()
    root = Path(__file__).resolve().parents[1]
    # a hardware queue for every slot's stream: in the default eight a small slot's kernels may stand
    # behind the large request's
    env = dict(os.environ, CUDA_DEVICE_MAX_CONNECTIONS="32")
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=root, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    lat = json.loads(r.stdout.strip().splitlines()[-1])
    # eight requests of a few milliseconds beside one of some hundreds
    assert max(lat["small"]) < 0.5 * lat["big"], lat
