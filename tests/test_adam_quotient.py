"""The quotient of the Adam update (csrc/mlp_kernels.cu) is the rounded one.

The function's own text is compiled for the host, where a / b rounds to nearest,
and compared bit for bit: dividends over the whole range where its remainder
does not underflow, signs, zeros, infinities and NaN; divisors 1 - beta^t.
"""
import ctypes as C
import os
import re
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = """
#include <cmath>
#define __device__
#define __forceinline__ inline
static inline float __fmul_rn(float a, float b) { return a * b; }
%s
extern "C" long long mismatches(const float* a, long long n, float b) {
  const float y = 1.0f / b;
  long long bad = 0;
  for (long long i = 0; i < n; i++) {
    const float q = quotient(a[i], b, y), w = a[i] / b;
    bad += !(q == w || (q != q && w != w));
  }
  return bad;
}
"""


def test_quotient_is_the_rounded_one(tmp_path):
    with open(os.path.join(ROOT, "paper_1702_04487_gb300", "csrc", "mlp_kernels.cu")) as fh:
        (text,) = re.findall(r"__device__ __forceinline__ float quotient\(.*?\n}\n", fh.read(), re.S)
    src, lib = tmp_path / "q.cpp", tmp_path / "q.so"
    src.write_text(SHIM % text)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", str(src), "-o", str(lib)],
                   check=True)
    f = C.CDLL(str(lib)).mismatches
    f.restype, f.argtypes = C.c_longlong, [C.c_void_p, C.c_longlong, C.c_float]
    rng = np.random.default_rng(1)
    a = np.ldexp(rng.integers(1 << 23, 1 << 24, 20000).astype(np.float64),
                 rng.integers(-99, 128, 20000) - 24)
    a = (a * rng.choice([-1, 1], a.size)).astype(np.float32)
    a = np.concatenate([a, np.array([0.0, -0.0, 1e-30, -1e-30, np.inf, -np.inf, np.nan,
                                     np.finfo(np.float32).max], np.float32)])
    for beta in (0.0, 0.5, 0.9, 0.95, 0.99, 0.999, 0.9999):
        for t in (1, 2, 3, 10, 100, 1000, 100000):
            b = np.float32(1) - np.power(np.float32(beta), np.float32(t))
            assert f(a.ctypes.data_as(C.c_void_p), a.size, b) == 0, (beta, t)
