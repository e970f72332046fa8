"""The float32-pair arithmetic of csrc/df.cuh, built by the host compiler (every operation is one IEEE-754 float32
operation, so that host and device agree bit for bit), against exact rational arithmetic."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "df.cuh"
using namespace rm;
extern "C" double sum_squares(const float* x, int n) {
    SumSq32 a;
    for (int i = 0; i < n; i++) a.add(x[i]);
    return a.value();
}
extern "C" float sum_floats(const float* x, int n) {
    CompSum a;
    for (int i = 0; i < n; i++) a.add(x[i]);
    return a.value();
}
extern "C" void convert(const double* x, int n, float* f, float* hi, float* lo) {
    for (int i = 0; i < n; i++) {   // each value beside its neighbours, as a thread converts them
        const double v[3] = {x[i], x[(i + 1) % n], x[(i + 41) % n]};
        float a[3], h[3], l[3];
        to_f32_n(v, a);
        df_split_n(v, h, l);
        f[i] = a[0];
        hi[i] = h[0];
        lo[i] = l[0];
    }
}
"""


@pytest.fixture(scope="module")
def df(tmp_path_factory):
    d = tmp_path_factory.mktemp("df")
    (d / "df.cpp").write_text(SRC)
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "tests", "fake", "host"), "-I",
                    os.path.join(ROOT, "paper_2112_04556_gb300", "csrc"), "-o", str(d / "df.so"), str(d / "df.cpp")],
                   check=True)
    L = ctypes.CDLL(str(d / "df.so"))
    L.sum_squares.restype = ctypes.c_double
    L.sum_floats.restype = ctypes.c_float
    return L


@pytest.mark.parametrize("n", [1, 2, 32, 448, 4096])
@pytest.mark.parametrize("spread", [0.0, 8.0, 30.0])
def test_sum_of_squares_is_float64_accurate(df, n, spread):
    """Sums of squares of one lane (448 terms: the largest lattice of the cooperative Krylov run; 4096: beyond any),
    normal values times 2^k, |k| <= spread (30: some squares leave float32's range and go through the float64 sum).  A
    float64 sum of n squares may be off by n 2^-53; this one by its last three additions and, where the float64 part
    holds some of the terms, theirs: 4 2^-53 and n 2^-53 of that part."""
    worst = 0.0
    for seed in range(20):
        rng = np.random.default_rng(seed)
        x = (rng.standard_normal(n) * 2.0 ** rng.uniform(-spread, spread, n)).astype(np.float32)
        got = df.sum_squares(x.ctypes.data_as(ctypes.c_void_p), n)
        want = sum(Fraction(float(v)) ** 2 for v in x)
        wide = sum(Fraction(float(v)) ** 2 for v in x if not 2.0 ** -40 <= abs(v) <= 2.0 ** 40)
        bound = (4 * want + n * wide) / 2 ** 53
        assert abs(Fraction(got) - want) <= bound, (seed, float(abs(Fraction(got) - want) / want))
        worst = max(worst, float(abs(Fraction(got) - want) / want))
    assert worst < 1e-12


def test_conversions_over_all_exponents(df):
    """to_f32 rounds as the conversion instruction does, subnormals, infinities and NaN included; df_split's pair holds a
    value to 2^-49 of it (2^-150 absolute among the subnormals), the high part a float next to it."""
    rng = np.random.default_rng(1)
    x = np.concatenate([((1.0 + rng.random(40)) * s * 2.0 ** e) for e in range(-1022, 1023) for s in (1, -1)])
    tie = np.float64(np.float32(1.0 + rng.random(200))) + 2.0 ** -24   # halves of a last place, either way
    x = np.concatenate([x, tie, -tie, tie * 2.0 ** -126, tie * 2.0 ** -127, [0.0, -0.0, 5e-324, np.inf, -np.inf, np.nan]])
    f, hi, lo = (np.empty(x.size, dtype=np.float32) for _ in range(3))
    ptr = [a.ctypes.data_as(ctypes.c_void_p) for a in (x, f, hi, lo)]
    df.convert(ptr[0], x.size, *ptr[1:])
    with np.errstate(over="ignore"):
        want = x.astype(np.float32)
    assert np.array_equal(f, want, equal_nan=True) and np.array_equal(np.signbit(f), np.signbit(want))
    ok = np.abs(x) < 2.0 ** 127
    h, l, v = hi[ok].astype(np.float64), lo[ok].astype(np.float64), x[ok]
    assert np.all(np.abs((v - h) - l) <= np.maximum(2.0 ** -49 * np.abs(v), 2.0 ** -150))
    assert np.all(np.abs(l) <= 0.5 * np.spacing(np.abs(hi[ok])).astype(np.float64))


@pytest.mark.parametrize("n", [1, 2, 14, 100])
def test_sums_of_a_lane_do_not_lose_with_their_length(df, n):
    """A lane's sum over its units, values of either sign: rounded once (2^-24 of the result) and n^2 2^-48 of the sum of
    the magnitudes (n errors of 2^-24 of partial sums, added up in float32), at any of the lengths a run has."""
    for seed in range(50):
        rng = np.random.default_rng(seed)
        x = (rng.standard_normal(n) * 2.0 ** rng.uniform(-6, 6, n)).astype(np.float32)
        got = Fraction(float(df.sum_floats(x.ctypes.data_as(ctypes.c_void_p), n)))
        want, size = sum(Fraction(float(v)) for v in x), sum(Fraction(abs(float(v))) for v in x)
        assert abs(got - want) <= abs(want) / 2 ** 24 + n * n * size / 2 ** 48
