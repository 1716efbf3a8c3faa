"""CPU test of what complex64 register phases take: builds ``rphase_plain_check.cpp`` against the
package's host sources with g++ and runs it."""
import shutil
import subprocess
from pathlib import Path

import pytest

from test_host_transforms_cpu import CSRC, ROOT, _cuda_include


def test_plain_phases_take_what_they_can(tmp_path):
    gxx, inc = shutil.which("g++"), _cuda_include()
    if gxx is None or inc is None or not any((Path(inc).parent / "lib64").glob("libcudart.so*")):
        pytest.skip("g++, the CUDA headers or the CUDA runtime library are not available")
    lib, exe = Path(inc).parent / "lib64", tmp_path / "rphase_plain_check"
    srcs = [ROOT / "tests" / "rphase_plain_check.cpp"] + \
        [CSRC / f for f in ("ir.cpp", "kgeom.cpp", "plan.cpp", "phasefn.cpp", "tpb.cpp", "rphase.cpp")]
    helpers = (ROOT / "tests" / "rphase_pack_check.cpp").read_text().split("\nint main(")[0]
    (tmp_path / "rphase_pack_helpers.h").write_text(helpers)
    cmd = [gxx, "-O1", "-std=c++17", f"-I{CSRC}", f"-I{ROOT / 'include'}", f"-I{inc}",
           f"-I{tmp_path}", f"-I{ROOT / 'tests'}", *map(str, srcs), f"-L{lib}", "-lcudart", f"-Wl,-rpath,{lib}",
           "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-4000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "OK" in r.stdout, r.stdout[-4000:]
