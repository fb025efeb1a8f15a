"""The resident CG's scalar steps (csrc/cg_scalars.cuh) run on the host: steps and
comparisons taken from FP32 pairs equal those of FP64 arithmetic on the doubles
the pairs stand for, at random and next to the ties and bounds."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = """
#include "cg_scalars.cuh"
using namespace hisq;
extern "C" void steps(long n, const double *a, const double *b, const double *den, float *out, float *pairs)
{
    for (long i = 0; i < n; i++) {
        out[i] = step_quotient(ff(a[i]), ff(b[i]), ff(den[i]), [&](double &x, double &y) {
            x = a[i] - b[i];
            y = den[i];
        });
        pairs[i] = ((ff(a[i]) - ff(b[i])) / ff(den[i])).hi;
    }
}
extern "C" void less(long n, const double *x, const double *y, int *out)
{
    for (long i = 0; i < n; i++)
        out[i] = decide_less(ff(x[i]).hi, ff(y[i]).hi, [&](double &u, double &v) { u = x[i], v = y[i]; });
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    from paper_2302_09224_gb300 import build

    d = tmp_path_factory.mktemp("scalars")
    src, lib = str(d / "s.cu"), str(d / "s.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc(), "-O2", "-std=c++17", "-shared", "--expt-relaxed-constexpr", "-Xcompiler",
                    "-fPIC,-ffp-contract=off", "-I" + build.CSRC, src, "-o", lib], check=True)
    return ctypes.CDLL(lib)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def steps(host, a, b, den):
    out, pairs = np.empty(a.size, np.float32), np.empty(a.size, np.float32)
    host.steps(ctypes.c_long(a.size), ptr(a), ptr(b), ptr(den), ptr(out), ptr(pairs))
    with np.errstate(all="ignore"):
        return out, pairs, ((a - b) / den).astype(np.float32)


def doubles(rng, n, lo, hi):
    return rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(lo, hi, n)


@pytest.mark.parametrize("lo,hi", [(-20, 20), (-90, -60), (-120, -70), (60, 100), (-110, 110)])
def test_random(host, lo, hi):
    rng = np.random.default_rng(1)
    n = 200000
    a, den = doubles(rng, n, lo, hi), doubles(rng, n, lo, hi)
    for b in (np.zeros(n), a * rng.normal(0, 1e-3, n), a * (1 - 2.0 ** -rng.integers(1, 50, n))):
        out, _, want = steps(host, a, b, den)
        assert np.array_equal(out, want)


def test_next_to_ties(host):
    """Quotients within 2^-52 to 2^-38 of a tie between two floats, the difference too."""
    rng = np.random.default_rng(2)
    n = 400000
    den = doubles(rng, n, -20, 20)
    f = rng.uniform(1.0, 2.0, n).astype(np.float32)
    tie = f.astype(np.float64) + 2.0 ** -24 * rng.choice([1.0, -1.0], n)
    q = tie * (1 + rng.choice([-1.0, 0.0, 1.0], n) * 2.0 ** -rng.integers(38, 54, n))
    a = q * den
    for b in (np.zeros(n), a * rng.normal(0, 1e-3, n), -7.5 * a):
        out, pairs, want = steps(host, a + b, b, den)
        assert np.array_equal(out, want)
        assert np.any(pairs != want)  # what the pairs alone would give


def test_comparisons(host):
    rng = np.random.default_rng(4)
    n = 400000
    x = np.concatenate([doubles(rng, n, -130, 120), doubles(rng, n, -10, 10), [0.0, 1e-300, 5e-324, 1e300]])
    y = x * (1 + rng.choice([-1.0, 0.0, 1.0], x.size) * 2.0 ** -rng.integers(0, 54, x.size).astype(np.float64))
    y[: n // 4] = doubles(rng, n // 4, -130, 120)
    out = np.empty(x.size, np.int32)
    host.less(ctypes.c_long(x.size), ptr(x), ptr(y), ptr(out))
    assert np.array_equal(out != 0, x < y)
