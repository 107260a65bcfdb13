"""Three-float arithmetic (csrc/tfl.h) on the CPU against exact rationals.

Bounds: each operation keeps the products and sums of its first two orders exactly and
rounds the third order (2^-48 of the result) to FP32, a handful of roundings: 2^-69 of the
product, 2^-70 of a sum's terms; the reciprocal root's last step squares an error of
2^-43 and doubles the product's: 2^-66."""
import ctypes
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2108_01786_gb300", "csrc", "tfl.h")
SRC = r"""
#include "%s"
static tfl ld(const float* v) { return {v[0], v[1], v[2]}; }
static void st(float* o, tfl v) { o[0] = v.s; o[1] = v.e; o[2] = v.f; }
extern "C" void mul(const float* a, const float* b, float* o) { st(o, ld(a) * ld(b)); }
extern "C" void sub(const float* a, const float* b, float* o) { st(o, ld(a) - ld(b)); }
extern "C" void root(const float* a, float x0, float* o) { st(o, tf_rsqrt_from(ld(a), x0)); }
extern "C" void sum(const float* v, int n, float* o) {
  tfl s = {0.f, 0.f, 0.f};
  for (int i = 0; i < n; ++i) { const tf_pair p = tf_two_prod(v[2 * i], v[2 * i + 1]); tf_add(s, p.h, p.l); }
  st(o, tf_norm(s));
}
"""


@pytest.fixture(scope="module")
def T(tmp_path_factory):
    d = tmp_path_factory.mktemp("tfl")
    src, so = str(d / "t.cpp"), str(d / "t.so")
    with open(src, "w") as f:
        f.write(SRC % HEADER)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-o", so, src], check=True)
    lib = ctypes.CDLL(so)

    def call(name, *args):
        o = np.zeros(3, dtype=np.float32)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p) if isinstance(a, np.ndarray) else a
        getattr(lib, name)(*[p(a) for a in args], p(o))
        return o
    return call


def _val(a):
    return sum((Fr(float(x)) for x in a), Fr(0))


def _draw(rng):
    v = rng.standard_normal() * 10.0 ** rng.uniform(-6, 6)
    h = np.float32(v)
    l = np.float32(v - np.float64(h))
    return np.array([h, l, np.float32(np.float64(l) * 2.0 ** -25 * rng.uniform(-1, 1))], dtype=np.float32)


def test_products_sums_and_roots(T):
    rng = np.random.default_rng(0)
    for _ in range(3000):
        a, b = _draw(rng), _draw(rng)
        va, vb = _val(a), _val(b)
        assert abs(_val(T("mul", a, b)) - va * vb) <= Fr(1, 2 ** 69) * abs(va * vb)
        assert abs(_val(T("sub", a, b)) - (va - vb)) <= Fr(1, 2 ** 70) * (abs(va) + abs(vb))
        a = a if a[0] > 0 else -a
        x0 = np.float32(1.0 / np.sqrt(np.float64(a[0])) * (1.0 + 2.0 ** -23 * rng.integers(-2, 3)))
        x = T("root", a, ctypes.c_float(float(x0)))
        assert abs(_val(a) * _val(x) ** 2 - 1) / 2 <= Fr(1, 2 ** 66)
        assert abs(x[1]) <= 2.0 ** -24 * abs(x[0]) * 1.001      # normalised
    zero = np.zeros(3, dtype=np.float32)
    assert not T("root", zero, ctypes.c_float(np.inf)).any()
    assert not T("root", np.array([-1, 0, 0], dtype=np.float32), ctypes.c_float(np.nan)).any()


@pytest.mark.parametrize("n", [1, 2, 31, 700, 5000])
def test_dots_beat_fp64(T, n):
    """Sums of products of floats, cancelling ones among them: within n 2^-71 of the sum of
    magnitudes, below FP64's n 2^-53."""
    rng = np.random.default_rng(n)
    v = rng.standard_normal((n, 2)).astype(np.float32)
    v[n // 2:, 0] = -v[:n - n // 2, 0]
    v[n // 2:, 1] = v[:n - n // 2, 1] * np.float32(1 + 2.0 ** -20)
    terms = [Fr(float(a)) * Fr(float(b)) for a, b in v]
    s = _val(T("sum", np.ascontiguousarray(v.reshape(-1)), ctypes.c_int(n)))
    assert abs(s - sum(terms)) <= Fr(n, 2 ** 71) * sum(abs(t) for t in terms)
