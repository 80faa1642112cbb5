"""The sums of the compensated phi accumulation (csrc/pair.cuh), compiled for the
host: phi + lo + (a + d) / 2 and / 6 as an FP32 pair.

Per sample the error against the exact sum is at most the rounding of the new low
part, half an ulp of it (2^-24 of it, or the smallest subnormal), plus the
terms dropped past the second order, 2^-70 of the largest summand.  Over all
samples it is no larger, in the mean square and at most, than that of the
same sum in FP64 stored as a pair."""
from __future__ import annotations

import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2011_00814_gb300", "csrc")
SRC = """
#include "pair.cuh"
extern "C" void run(int six, long long n, const float* ph, const float* lo, const float* a, const float* d, float* hi,
                    float* low) {
  for (long long i = 0; i < n; ++i) {
    if (six) gpe2p::pair_sixth(ph[i], lo[i], a[i], d[i], hi[i], low[i]);
    else gpe2p::pair_half(ph[i], lo[i], a[i], d[i], hi[i], low[i]);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("pair")
    (d / "pair.cpp").write_text(SRC)
    so = str(d / "pair.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, "-o", so,
                    str(d / "pair.cpp")], check=True)
    return ctypes.CDLL(so)


def samples(n, seed, phi):
    rng = np.random.default_rng(seed)
    if phi == "bulk":      # phi near +-1, steps of the method
        ph = rng.choice([-1.0, 1.0], n) * (1.0 + 1e-2 * rng.standard_normal(n))
    elif phi == "any":
        ph = rng.uniform(-1.2, 1.2, n)
    else:                  # the interface, phi smaller than its increment
        ph = rng.uniform(-1, 1, n) * 10.0 ** rng.uniform(-9, 0, n)
    ph = ph.astype(np.float32)
    lo = (rng.uniform(-0.5, 0.5, n) * np.spacing(np.abs(ph))).astype(np.float32)
    a, d = ((rng.uniform(-1, 1, n) * 10.0 ** rng.uniform(-9, 0, n)).astype(np.float32) for _ in range(2))
    return ph, lo, a, d


@pytest.mark.parametrize("phi", ["bulk", "any", "small"])
@pytest.mark.parametrize("six", [0, 1])
def test_pair_is_as_exact_as_an_fp64_sum(lib, six, phi):
    n = 100000
    ph, lo, a, d = samples(n, 3 + six, phi)
    hi, low = np.empty(n, np.float32), np.empty(n, np.float32)
    p = lambda x: x.ctypes.data_as(ctypes.POINTER(ctypes.c_float))
    lib.run(six, ctypes.c_longlong(n), p(ph), p(lo), p(a), p(d), p(hi), p(low))
    s = a.astype(np.float64) + d.astype(np.float64)
    pn = ph.astype(np.float64) + lo.astype(np.float64)
    o = pn + s * (1.0 / 6.0) if six else pn + 0.5 * s
    hi64 = o.astype(np.float32)
    low64 = (o - hi64.astype(np.float64)).astype(np.float32)

    def errors(h, l):  # c times the error of the pair, exactly rounded
        c = 6.0 if six else 2.0
        rows = zip(*(x.astype(np.float64) for x in (c * ph.astype(np.float64), c * lo.astype(np.float64), a, d,
                                                    -c * h.astype(np.float64), -c * l.astype(np.float64))))
        return np.array([math.fsum(r) for r in rows]) / c

    e, e64 = errors(hi, low), errors(hi64, low64)
    big = np.maximum(np.maximum(np.abs(ph), np.abs(a)), np.abs(d)).astype(np.float64)
    assert np.all(np.abs(e) <= 2.0 ** -24 * np.abs(low.astype(np.float64)) + 2.0 ** -70 * big + 2.0 ** -150)
    assert np.sqrt(np.mean(e ** 2)) <= np.sqrt(np.mean(e64 ** 2)) * 1.0001
    assert np.max(np.abs(e)) <= np.max(np.abs(e64)) * 1.0001
