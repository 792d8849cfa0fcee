"""Sum of FP32 pairs in the fused loops (csrc/sum3.h), on the host: as precise as FP64 additions.

The pairs are block partials hi + lo with |lo| at most half a unit of hi.  In lanes of five and a tree
of 32, as the loops take them, the result differs from the exact sum by half an FP64 unit of it and by
what the third terms lose: at most 304 of them, of 2^-48 of the sum of magnitudes each, rounded to
2^-24 of that: 2^-63 of the sum of magnitudes.  (A double-float sum is off by up to some 2^-46.)
"""
import ctypes as C
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2510_09812_gb300", "csrc")
SRC = """
#include "sum3.h"
extern "C" double sum3(int n, const float* h, const float* l) {
  gspm::Sum3 t[32];
  for (int k = 0; k < n; ++k) t[k % 32].add(h[k], l[k], 0.f);
  for (int o = 16; o >= 1; o >>= 1)
    for (int i = 0; i < o; ++i) t[i].add(t[i + o].s, t[i + o].e, t[i + o].f);
  return t[0].value();
}
"""


@pytest.fixture(scope="module")
def sum3(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("sum3")
    (d / "s.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    "-o", str(d / "s.so"), str(d / "s.cpp")], check=True)
    f = C.CDLL(str(d / "s.so")).sum3
    f.restype = C.c_double
    f.argtypes = [C.c_int, C.c_void_p, C.c_void_p]
    return lambda h, l: f(len(h), h.ctypes.data, l.ctypes.data)


@pytest.mark.parametrize("n", [1, 2, 31, 33, 152, 160])
@pytest.mark.parametrize("kind", ["positive", "signed", "spread", "cancelling", "zero"])
def test_as_precise_as_fp64(sum3, n, kind):
    rng = np.random.default_rng(n)
    for _ in range(50):
        x = {"positive": rng.random(n), "signed": rng.standard_normal(n),
             "spread": rng.standard_normal(n) * 10.0 ** rng.uniform(-12, 12, n),
             "cancelling": np.concatenate([rng.standard_normal((n + 1) // 2)] * 2)[:n]
             * np.where(np.arange(n) < (n + 1) // 2, 1.0, -1.0 - 1e-9),
             "zero": np.zeros(n)}[kind]
        h = x.astype(np.float32)
        l = (x - h).astype(np.float32)
        terms = [Fraction(float(a)) + Fraction(float(b)) for a, b in zip(h, l)]
        exact = sum(terms)
        size = sum(abs(t) for t in terms)
        off = abs(Fraction(sum3(h, l)) - exact)
        assert off <= abs(exact) * Fraction(1, 2 ** 53) + size * Fraction(1, 2 ** 63)
