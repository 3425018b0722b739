"""Particles per CTA of the fine stage (csrc/fine_choice.h), compiled for the
host: CTAs whose places mostly hold no particle are not chosen where smaller
ones leave fewer waves of work (no GPU needed)."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def choice(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("fine")
    src = d / "fine.cpp"
    src.write_text('#include "fine_choice.h"\nextern "C" int choice(int tiles, int ne, int sms, int per_sm1)\n'
                   "{ return iewpf::qhalf::fine_choice([&](int n) { return (long long)tiles * ((ne + n - 1) / n); },"
                   " sms, per_sm1); }\n")
    so = d / "fine.so"
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1910_01031_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    return lambda nx, ny, ne, sms=152, per_sm1=4: L.choice(-(-nx // 64) * -(-ny // 32), ne, sms, per_sm1)


@pytest.mark.parametrize("n", [64, 256, 512, 1000, 1024, 2048, 4096])
def test_few_particles_do_not_take_large_ctas(choice, n):
    """From a wave of CTAs on, 16 places for up to 4 particles take more than twice the time of 4."""
    for ne in (1, 2, 3, 4):
        assert choice(n, n, ne) < 16, ne
        assert choice(n, n, ne, per_sm1=2) < 16, ne
    assert choice(n, n, 1) == 1


def test_large_ensembles_take_16_and_small_problems_1(choice):
    for nx, ny, ne in ((512, 512, 100), (624, 624, 1000), (1024, 1024, 256), (1024, 1024, 16), (256, 256, 100)):
        assert choice(nx, ny, ne) == 16
    for nx, ny, ne in ((64, 64, 10), (48, 48, 4), (256, 256, 9), (512, 512, 2)):
        assert choice(nx, ny, ne) == 1
    for nx, ny, ne in ((512, 512, 8), (1024, 1024, 4), (1024, 1024, 8), (256, 256, 30)):
        assert choice(nx, ny, ne) == 4
