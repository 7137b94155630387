"""The stack rule of the cooperative walks, compiled for the host: no depth,
no width of a round and no share of children kept outgrows the stack."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    out = str(tmp_path_factory.mktemp("walk_take") / "walk_take.so")
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-fPIC", "-shared", "-I", os.path.join(ROOT, "tests", "host_emu"),
                        "-I", os.path.join(ROOT, "paper_2605_01919_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "host_emu", "walk_take_host.cpp"), "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(out).walk_take_host


# (capacity, entries a round) of the warp walks, of the packet and coverage
# walks (no room beyond 448 and 512) and of the insertion's warps and blocks.  A
# rule without the reserve for the depth needs 521 of 520 entries at (512, 32) on
# 7 levels, which the tangent and scored walks had.
@pytest.mark.parametrize("cap, width", [(581, 32), (440, 4), (504, 4), (2048, 32), (8192, 256)])
def test_stack_never_outgrown(host, cap, width):
    reserve = ctypes.c_int()
    for levels in range(1, 13):
        for keep in (256, 250, 230, 200, 128):
            most = host(levels, cap, width, keep, 20000, 7 * levels + keep, ctypes.byref(reserve))
            assert 0 < most <= cap + reserve.value, (levels, keep, most)
