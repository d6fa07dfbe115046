"""QSum (metric_q.cuh), the exact sum of FP32 Q sums, compiled for the host: it
equals the exact rational sum for every multiple of 2^-77 below 2^20, the small
remainders included that nearly cancelling windows of one slot leave."""
import ctypes
import os
import random
import struct
import subprocess
from fractions import Fraction

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1803_00737_gb300", "csrc")
SRC = r"""
#include <cstdint>
#include <cstring>
#define __host__
#define __device__
#define __forceinline__ inline
static inline uint32_t __float_as_uint(float f) { uint32_t w; std::memcpy(&w, &f, 4); return w; }
static inline long long __shfl_xor_sync(unsigned, long long v, int) { return v; }
#include "metric_q.cuh"
extern "C" void qsum(const float *q, int n, long long *out) {
    dwtfuse::QSum s;
    for (int i = 0; i < n; ++i) s.add(q[i]);
    out[0] = s.hi;
    out[1] = s.lo;
}
"""


@pytest.fixture(scope="module")
def qsum(tmp_path_factory):
    d = tmp_path_factory.mktemp("qsum")
    (d / "q.cpp").write_text(SRC)
    so = str(d / "q.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "q.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def call(values):
        a = (ctypes.c_float * len(values))(*values)
        out = (ctypes.c_longlong * 2)()
        lib.qsum(a, len(values), out)
        return Fraction(out[0], 2 ** 32) + Fraction(out[1], 2 ** 77)

    return call


def _f32(x):
    return struct.unpack("f", struct.pack("f", x))[0]


def test_edges(qsum):
    for v in (0.0, -0.0, 1.0, -1.0, 2.0 ** -32, 2.0 ** -33, 2.0 ** -53, 2.0 ** -54, 2.0 ** -55, -(2.0 ** -60),
              2.0 ** -77, -(2.0 ** -77), 3 * 2.0 ** -77, 2.0 ** 20 - 0.0625, _f32(0.1), -_f32(1e-9)):
        assert qsum([v]) == Fraction(v), v


def test_random_sums(qsum):
    rng = random.Random(3)
    for _ in range(200):
        values = []
        for _ in range(64):
            m, e = rng.getrandbits(24), rng.randint(-77, -4)
            values.append(rng.choice((-1, 1)) * m * 2.0 ** e)
        assert all(_f32(v) == v for v in values)
        assert qsum(values) == sum(map(Fraction, values))
