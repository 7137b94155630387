"""The cull's workspace: bounded, a part of the free memory, and smaller when
the device refuses it (a fake device on the CPU)."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    out = str(tmp_path_factory.mktemp("chunk") / "chunk.so")
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-fPIC", "-shared",
                        "-I", os.path.join(ROOT, "paper_2605_01919_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "host_emu", "chunk_host.cpp"), "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(out)
    L.chunk_host.argtypes = [ctypes.c_longlong] * 3
    L.chunk_host.restype = ctypes.c_longlong
    L.shrink_host.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    L.shrink_host.restype = ctypes.c_longlong
    return L


@pytest.mark.parametrize("tiles, per, free", [(1, 1536, 1 << 38), (8192, 642 * 128, 1 << 38), (1 << 20, 642 * 128, 1 << 38),
                                              (8192, 642 * 128, 1 << 30), (8192, 642 * 128, 0), (3, 40962 * 128, 1 << 20)])
def test_chunk_bounds(lib, tiles, per, free):
    c = lib.chunk_host(tiles, per, free)
    assert 1 <= c <= tiles
    assert c == 1 or c * per <= min(17 << 26, free // 8)
    assert c == tiles or (c + 1) * per > min(17 << 26, free // 8)


@pytest.mark.parametrize("size, fits", [(8192, 8192), (8192, 8191), (8192, 100), (7, 1), (1, 1)])
def test_a_refused_workspace_is_halved_until_it_fits(lib, size, fits):
    tried = ctypes.c_int()
    got = lib.shrink_host(size, fits, 0, ctypes.byref(tried))
    assert 1 <= got <= fits and (got == size or 2 * got > fits - 1)
    assert tried.value == (size // got).bit_length() or size >> (tried.value - 1) == got


def test_no_room_at_all_and_other_errors_are_reported(lib):
    tried = ctypes.c_int()
    assert lib.shrink_host(8192, 0, 0, ctypes.byref(tried)) == -2 and tried.value == 14
    assert lib.shrink_host(8192, 10, 3, ctypes.byref(tried)) == -3 and tried.value == 3
