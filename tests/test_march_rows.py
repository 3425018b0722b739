"""Chunk lengths that the tuner of the scheme step tries (csrc/march_rows.h),
compiled for the host: on every grid height there is one near each length that
a problem may want, from all rows down to what many short chunks need (no GPU
needed)."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def march_rows(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rows")
    src = d / "rows.cpp"
    src.write_text('#include "march_rows.h"\nextern "C" int rows(int ny, int* out)\n'
                   "{ const auto th = iewpf::march_rows(ny); for (int t : th) *out++ = t; return (int)th.size(); }\n")
    so = d / "rows.so"
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1910_01031_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))

    def rows(ny):
        out = (ctypes.c_int * 64)()
        return list(out[:L.rows(ny, out)])
    return rows


@pytest.mark.parametrize("ny", [15, 16, 17, 48, 64, 65, 100, 300, 341, 512, 624, 700, 1000, 1024, 2048, 4096])
def test_lengths_are_equal_chunks_close_to_every_wanted_length(march_rows, ny):
    th = march_rows(ny)
    assert th[0] == ny and th == sorted(set(th), reverse=True) and th[-1] >= 2
    for t in th:
        assert -(-ny // -(-ny // t)) == t           # the longest chunk of that many equal ones
    want = 16
    while want <= ny:
        # within the square root of the largest step between candidates (2, 3/2 from the second on) and rounding up
        assert any(t <= 1.42 * want and want <= 1.42 * t for t in th), (want, th)
        want *= 2
    # as many chunks as lengths of 16, 32, ... rows make
    for t in (16, 32, 64, 128, 256, 512):
        if t <= ny:
            n = -(-ny // t)
            assert -(-ny // n) in th
