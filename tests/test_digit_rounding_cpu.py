"""split_times_pow2 (tc_ptx.cuh), the last step of every tensor-core FP64 product: the
exact digit sum (T 2^32 + r) 2^e rounded once to FP64, against Python's correctly rounded
integer division.  Exact equality: ties, both signs, zero words, the subnormal range and
both of its ends, overflow."""
import ctypes as C
import math
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "tc_ptx.cuh"
extern "C" double rounded(long long T, unsigned int r, int e) { return dqmc::split_times_pow2(T, r, e); }
"""


@pytest.fixture(scope="module")
def rounded(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("rounding")
    (d / "r.cu").write_text(SRC)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-I", os.path.join(ROOT, "paper_2003_05286_gb300", "csrc"), str(d / "r.cu"), "-o",
                    str(d / "r.so")], check=True)
    f = C.CDLL(str(d / "r.so")).rounded
    f.argtypes, f.restype = [C.c_longlong, C.c_uint, C.c_int], C.c_double
    return f


def _want(T, r, e):
    n = (T << 32) + r
    try:
        return float(n << e) if e >= 0 else n / (1 << -e)     # int / int rounds once
    except OverflowError:
        return math.copysign(math.inf, n)


def _sums(rng, count):
    for _ in range(count):
        n = rng.getrandbits(rng.randint(1, 94))
        kind = rng.randint(0, 3)
        if kind == 1:                                          # a tie, or one beside it
            n = (rng.getrandbits(53) | (1 << 52)) << rng.randint(1, 40)
            n += rng.choice((-1, 0, 1)) + (1 << rng.randint(0, 40))
        elif kind == 2:                                        # runs of ones: carries
            n = ((1 << rng.randint(1, 93)) - 1) << rng.randint(0, 10)
        n = min(n, (1 << 94) - 1) * rng.choice((-1, 1))
        yield n >> 32, n & 0xFFFFFFFF, max(n.bit_length(), 1)


@pytest.mark.parametrize("top", ["normal", "subnormal", "smallest", "largest"])
def test_rounded_once(rounded, top):
    rng = random.Random(5)
    for T, r, bits in _sums(rng, 20000):
        # the exponent of the leading bit
        lead = {"normal": rng.randint(-1000, 1000), "subnormal": rng.randint(-1074, -1018),
                "smallest": rng.randint(-1080, -1070), "largest": rng.randint(1020, 1026)}[top]
        e = lead - (bits - 1)
        got, want = rounded(T, r, e), _want(T, r, e)
        assert got == want and math.copysign(1.0, got) == math.copysign(1.0, want if want else (-1.0 if T < 0 else 1.0)), (T, r, e)


def test_zero(rounded):
    for e in (-2000, -72, 0, 2000):
        assert rounded(0, 0, e) == 0.0
