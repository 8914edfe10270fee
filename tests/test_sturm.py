"""The eigenvalue counts of csrc/sturm.cuh, compiled for the host, where the
tridiagonal matrix decouples and the point is an eigenvalue exactly: the count
lies between the eigenvalues below the point and those not above it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01480_gb300", "csrc")

SOURCE = r"""
#include <math.h>
#include <string.h>
#include <algorithm>
#include <vector>
#define __device__
#define __forceinline__ inline
struct float2 { float x, y; };
struct float4 { float x, y, z, w; };
static float2 make_float2(float x, float y) { return {x, y}; }
static unsigned __float_as_uint(float f) { unsigned u; memcpy(&u, &f, 4); return u; }
static float __uint_as_float(unsigned u) { float f; memcpy(&f, &u, 4); return f; }
static unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return (hi << s) | (lo >> (32 - s)); }
static int __popc(unsigned x) { return __builtin_popcount(x); }
#include "sturm.cuh"

extern "C" void counts(const float* d, const float* e, int k, const float* x, int n, int* one, int* two) {
  const int groups = (k + 2) / 4;
  std::vector<float2> buf(1 + 4 * groups + 2);
  for (int i = 0; i < 1 + 4 * groups; ++i)
    buf[i] = i < k ? ttr::sturm_row(d[i], i > 0 ? e[i - 1] : 0.f) : ttr::sturm_row(16.f, 0.f);
  for (int j = 0; j < n; ++j) {
    int c0, c1;
    one[j] = ttr::sturm(buf.data(), groups, x[j]);
    ttr::sturm2(buf.data(), groups, x[j], x[n - 1 - j], c0, c1);
    two[j] = c0;
  }
}
"""


@pytest.fixture(scope="module")
def counts(tmp_path_factory):
    d = tmp_path_factory.mktemp("sturm")
    src, so = d / "sturm.cpp", d / "sturm.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))

    def run(d, e, x):
        d, e, x = (np.ascontiguousarray(a, dtype=np.float32) for a in (d, e, x))
        one, two = np.zeros(len(x), np.int32), np.zeros(len(x), np.int32)
        ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        lib.counts(ptr(d), ptr(e), len(d), ptr(x), len(x), ptr(one), ptr(two))
        assert (one == two).all()
        return one
    return run


def _check(counts, d, e):
    T = np.diag(np.float64(d)) + np.diag(np.float64(e), 1) + np.diag(np.float64(e), -1)
    lam = np.linalg.eigvalsh(T)
    x = np.unique(np.float32(np.concatenate([lam, d, np.linspace(-2.1, 2.1, 97)])))
    got = counts(d, e, x)
    # off-diagonals of 2^-30 move an eigenvalue by that much at most; 1e-6 also
    # covers the counts' own rounding
    below = (lam[None, :] < np.float64(x)[:, None] - 1e-6).sum(1)
    upto = (lam[None, :] <= np.float64(x)[:, None] + 1e-6).sum(1)
    assert (got >= below).all() and (got <= upto).all()


def test_diagonal_after_an_exact_hit(counts):
    d = np.float32([1, .5, .5, .5, .5, .25, .25, 0, 0, 0, 0])
    assert counts(d, np.zeros(10), [1.0])[0] >= 10
    _check(counts, d, np.zeros(10, np.float32))


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 8, 9, 33, 150])
def test_decoupled_and_coupled_matrices(counts, k):
    rng = np.random.default_rng(k)
    for _ in range(40):
        d = np.float32(rng.integers(-8, 9, k) / 8)
        _check(counts, d, np.zeros(max(0, k - 1), np.float32))
        e = np.float32(rng.integers(0, 3, max(0, k - 1)) / 4 * (rng.random(max(0, k - 1)) < 0.5))
        _check(counts, d, e)
        _check(counts, np.float32(rng.uniform(-1, 1, k)), np.float32(rng.uniform(0, 0.5, max(0, k - 1))))
