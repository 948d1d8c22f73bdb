"""Sums in three floats (csrc/float_sum.cuh) against the exact sum, and against FP64 sums (CPU).

The kernels that add FP32 shares and terms this way replace FP64 additions, so the error may not
exceed theirs.  Every addition rounds at 2^-72 of the largest partial sum at most (three roundings
of 2^-24 nested), and get() rounds twice in FP64.
"""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1305_4196_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("float_sum")
    src, so = d / "s.cpp", d / "s.so"
    src.write_text("""#include "float_sum.cuh"
extern "C" {
double sum(const float* x, long n) { mdgb::FloatSum s; for (long i = 0; i < n; ++i) s.add(x[i]); return s.get(); }
// n numbers in `lanes` sums, added by a butterfly; the results of all lanes
void butterfly(const float* x, long n, int lanes, double* out) {
    mdgb::FloatSum s[64];
    for (long i = 0; i < n; ++i) s[i % lanes].add(x[i]);
    for (int o = 1; o < lanes; o <<= 1) {
        mdgb::FloatSum t[64];
        for (int l = 0; l < lanes; ++l) t[l] = s[l], t[l].add(s[l ^ o]);
        for (int l = 0; l < lanes; ++l) s[l] = t[l];
    }
    for (int l = 0; l < lanes; ++l) out[l] = s[l].get();
}
}
""")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    L = C.CDLL(str(so))
    L.sum.restype = C.c_double
    L.sum.argtypes = [C.c_void_p, C.c_long]
    L.butterfly.argtypes = [C.c_void_p, C.c_long, C.c_int, C.c_void_p]
    return L


def _inputs(kind, n, rng):
    x = rng.normal(size=n) * 10.0 ** rng.uniform(-6, 6, n) if kind == "wide" else rng.normal(size=n)
    if kind == "cancelling":  # pairs of opposite numbers around small ones
        x[: n // 2] = 1e6 * rng.normal(size=n // 2)
        x[n // 2: n // 2 * 2] = -x[: n // 2]
        x = np.append(rng.permutation(x), 1e-3 * rng.normal(size=5))
    if kind == "one sign":
        x = np.abs(x) + 0.5
    return x.astype(np.float32)


@pytest.mark.parametrize("kind", ["plain", "one sign", "wide", "cancelling"])
@pytest.mark.parametrize("n", [1, 2, 14, 76, 4096])
def test_sum_is_no_less_exact_than_fp64(lib, kind, n):
    rng = np.random.default_rng(n)
    worst = worst64 = 0.0
    for _ in range(50):
        x = np.ascontiguousarray(_inputs(kind, n, rng))
        exact = math.fsum(x.tolist())
        partial = float(np.max(np.abs(np.cumsum(x.astype(np.float64)))))
        bound = 2.0 ** -53 * (2.0 * abs(exact)) + len(x) * 2.0 ** -72 * partial * 4
        got = lib.sum(x.ctypes.data, len(x))
        assert abs(got - exact) <= bound
        fp64 = float(np.cumsum(x.astype(np.float64))[-1])
        worst, worst64 = max(worst, abs(got - exact)), max(worst64, abs(fp64 - exact))
        out = np.empty(32)
        lib.butterfly(x.ctypes.data, len(x), 32, out.ctypes.data)
        # (the lanes' partial sums can be as large as all terms of one sign together)
        scale = float(np.abs(x.astype(np.float64)).sum())
        assert (out == out[0]).all() and abs(out[0] - exact) <= 2.0 ** -53 * 2.0 * abs(exact) + len(x) * 2.0 ** -70 * scale
    assert worst <= worst64 + 2.0 ** -53 * abs(exact)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_what_is_not_finite_is_seen(lib, bad):
    x = np.ones(40, dtype=np.float32)
    x[17] = bad
    assert not math.isfinite(lib.sum(x.ctypes.data, 40))
    big = np.full(3, 3.0e38, dtype=np.float32)  # finite in FP64, beyond FP32
    assert not math.isfinite(lib.sum(big.ctypes.data, 3))
