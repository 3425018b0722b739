"""The two-float logarithm of the random vectors' uniforms (csrc/log_uniform.h),
compiled for the host, where it gives the device's bits (every operation is
IEEE), against the long double logarithm (no GPU needed)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def log_uniform(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("log")
    src = d / "log.cpp"
    src.write_text('#include "log_uniform.h"\nextern "C" void logs(const uint32_t* a, long n, float* hi, float* lo)\n'
                   "{ for (long i = 0; i < n; ++i) iewpf::log_uniform(a[i], hi[i], lo[i]); }\n")
    so = d / "log.so"
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1910_01031_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))

    def logs(a):
        a = np.ascontiguousarray(a, np.uint32)
        hi, lo = np.empty(a.size, np.float32), np.empty(a.size, np.float32)
        vp = ctypes.c_void_p
        L.logs(a.ctypes.data_as(vp), ctypes.c_long(a.size), hi.ctypes.data_as(vp), lo.ctypes.data_as(vp))
        return hi, lo
    return logs


def _exact(a):
    a = a.astype(np.int64)
    scale = np.longdouble(2) ** -33
    return np.where(a < 2 ** 31, np.log((2 * a + 1).astype(np.longdouble) * scale),
                    np.log1p(-(2 * (2 ** 32 - 1 - a) + 1).astype(np.longdouble) * scale))


def _inputs(name):
    rng = np.random.default_rng(5)
    if name == "random":
        return rng.integers(0, 2 ** 32, 1 << 20)
    small = np.floor(2.0 ** (32 * rng.random(1 << 18))).astype(np.int64)
    if name == "next to 0":
        return np.concatenate([np.arange(4096), small])
    if name == "next to 1":
        return 2 ** 32 - 1 - np.concatenate([np.arange(4096), small])
    # powers of two, where the exponent changes, and their multiples by sqrt(1/2), where the reduction does
    p = 2 ** np.arange(1, 33, dtype=np.int64)
    r = (p * np.sqrt(0.5)).astype(np.int64)
    return np.clip(np.concatenate([v + d for v in (p, r, np.array([0xB504F334])) for d in range(-3, 4)]), 0, 2 ** 32 - 1)


@pytest.mark.parametrize("name", ["random", "next to 0", "next to 1", "edges"])
def test_relative_error_is_below_2_to_minus_28(log_uniform, name):
    a = _inputs(name)
    hi, lo = log_uniform(a)
    ref = _exact(a)
    # the low word is what rounding to float leaves
    assert (np.abs(lo) <= np.abs(hi) * np.float32(2.0 ** -24)).all()
    rel = np.abs((hi.astype(np.longdouble) + lo - ref) / ref)
    assert float(rel.max()) < 2.0 ** -28


def test_products_round_to_float_as_those_of_double_logarithms(log_uniform):
    """r^2 of a pair of uniforms as the random vectors form it: at most one unit in the last place off, and mostly
    the bits, of the product of FP64 logarithms rounded to float (a relative error of 2^-30 in the mean moves
    a rounding of 2^-24 in fewer than one of 16 cases)."""
    a, b = _inputs("random"), np.random.default_rng(6).integers(0, 2 ** 32, 1 << 20)
    (xh, xl), (nh, nl) = log_uniform(a), log_uniform(b)
    f32, f64 = np.float32, np.float64
    q = xh * nh
    e = (xh.astype(f64) * nh - q).astype(f32) + (xh.astype(f64) * nl + (xl * nh)).astype(f32)
    got = f32(4) * (q + e)
    ref = (4 * _exact(a).astype(f64) * _exact(b).astype(f64)).astype(f32)
    assert (np.abs(got - ref) <= np.spacing(ref)).all()
    assert np.mean(got != ref) < 2.0 ** -4
