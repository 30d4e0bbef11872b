"""Waves of a batch's shares (csrc/fq_shares.h, compiled for the host): more than
one where shares within runs leave warps idle, and then less time by the shares'
own measure."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2601_19505_gb300", "csrc")
WRAP = """
#include "fq_shares.h"
static std::vector<fq::ShareRun> runs(unsigned n, const unsigned* B, const double* fill) {
    std::vector<fq::ShareRun> v;
    for (unsigned i = 0; i < n; ++i) v.push_back({B[i], fill[i]});
    return v;
}
extern "C" unsigned waves(unsigned n, const unsigned* B, const double* fill, unsigned nw) {
    return fq::share_waves(runs(n, B, fill), nw);
}
extern "C" double bound(unsigned n, const unsigned* B, const double* fill, unsigned nw) {
    return fq::share_bound(runs(n, B, fill), nw);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("waves")
    (d / "wrap.cpp").write_text(WRAP)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "wrap.cpp"),
                    "-o", str(d / "libwaves.so")], check=True)
    L = ctypes.CDLL(str(d / "libwaves.so"))
    L.bound.restype = ctypes.c_double
    return L


def _args(n, B, fill):
    B = np.full(n, B, dtype=np.uint32) if np.isscalar(B) else np.asarray(B, dtype=np.uint32)
    fill = np.full(n, fill, dtype=np.float64) if np.isscalar(fill) else np.asarray(fill, dtype=np.float64)
    return (B, fill), (ctypes.c_uint(n), B.ctypes.data_as(ctypes.c_void_p),
                       fill.ctypes.data_as(ctypes.c_void_p))


@pytest.mark.parametrize("n,B,want", [(2, 340, 1), (3, 2432, 1), (64, 68, 1), (810, 68, 1), (1216, 68, 1),
                                      (1024, 68, 3), (1900, 68, 4), (2432, 68, 1), (1900, 1, 1)])
def test_equal_runs(lib, n, B, want):
    keep, a = _args(n, B, 159.0)
    assert lib.waves(*a, ctypes.c_uint(2432)) == want


@pytest.mark.parametrize("seed", range(20))
def test_waves_are_worth_it(lib, seed):
    rng = np.random.default_rng(seed)
    n = int(np.exp(rng.uniform(np.log(2.0), np.log(4000.0))))
    keep, a = _args(n, rng.integers(1, 400, n), rng.uniform(30.0, 180.0, n))
    for nw in (1216, 2432, 3648):
        if nw < n:
            continue
        t = [k * (lib.bound(*a, ctypes.c_uint(k * nw)) + 100.0) for k in (1, 2, 3, 4)]
        k = lib.waves(*a, ctypes.c_uint(nw))
        assert k == 1 and min(t) >= t[0] / 1.05 or k > 1 and t[k - 1] == min(t[1:]) < t[0] / 1.05
