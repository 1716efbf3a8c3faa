"""CPU test of register phases in layers (``rphase.cpp``): builds ``rphase_pack_check.cpp``
against the package's host sources with g++ and runs it on seeded random circuits.  Phases must
act as their circuit, every phase in layers as the phase it was made from (to 1e-12, in double
precision), within the limits the kernel relies on."""
import shutil
import subprocess
from pathlib import Path

import pytest

from test_host_transforms_cpu import CSRC, ROOT, _cuda_include


@pytest.mark.parametrize("seed", [1, 2])
def test_layers_act_as_the_phase(seed, tmp_path):
    gxx, inc = shutil.which("g++"), _cuda_include()
    if gxx is None or inc is None or not any((Path(inc).parent / "lib64").glob("libcudart.so*")):
        pytest.skip("g++, the CUDA headers or the CUDA runtime library are not available")
    lib, exe = Path(inc).parent / "lib64", tmp_path / "rphase_pack_check"
    srcs = [ROOT / "tests" / "rphase_pack_check.cpp"] + \
        [CSRC / f for f in ("ir.cpp", "kgeom.cpp", "plan.cpp", "phasefn.cpp", "tpb.cpp", "rphase.cpp")]
    cmd = [gxx, "-O1", "-std=c++17", f"-I{CSRC}", f"-I{ROOT / 'include'}", f"-I{inc}", *map(str, srcs),
           f"-L{lib}", "-lcudart", f"-Wl,-rpath,{lib}", "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-4000:]
    r = subprocess.run([str(exe), str(seed), "2"], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "OK" in r.stdout, r.stdout[-4000:]
