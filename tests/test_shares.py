"""The shares of a batch's segments (csrc/fq_shares.h), compiled for the host:
every segment belongs to exactly one warp, a share lies within one run, and
there are never more shares than warps."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2601_19505_gb300", "csrc")
WRAP = """
#include "fq_shares.h"
extern "C" int cuts(unsigned n, const unsigned* B, const double* fill, unsigned nw, unsigned* out) {
    std::vector<fq::ShareRun> runs;
    for (unsigned i = 0; i < n; ++i) runs.push_back({B[i], fill[i]});
    std::vector<unsigned> c;
    if (!fq::share_cuts(runs, nw, c)) return 0;
    for (unsigned i = 0; i <= nw; ++i) out[i] = c[i];
    return c.size() == (size_t)nw + 1;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("shares")
    (d / "wrap.cpp").write_text(WRAP)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    str(d / "wrap.cpp"), "-o", str(d / "libshares.so")], check=True)
    return ctypes.CDLL(str(d / "libshares.so"))


def _cuts(lib, B, fill, nw):
    B = np.ascontiguousarray(B, dtype=np.uint32)
    fill = np.ascontiguousarray(fill, dtype=np.float64)
    out = np.zeros(nw + 1, dtype=np.uint32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    ok = lib.cuts(len(B), p(B), p(fill), nw, p(out))
    return out if ok else None


def _check(cuts, B):
    cuts = cuts.astype(np.int64)
    ends = np.cumsum(np.asarray(B, dtype=np.int64))
    assert cuts[0] == 0 and cuts[-1] == ends[-1]
    assert np.all(np.diff(cuts) >= 0)
    # a share holds no run's last segment together with the next run's first
    assert np.isin(ends, cuts).all()


# segments and expected spawns a segment of runs of 5e3, 1e4, 2e4, 172137.56 and
# 1e6 walkers on 152 SMs: floor(B w / w) of the first four is B - 1 for w = 32 + fill
SIZES = [(172, 1.1 * 5e3 / 172), (344, 1.1 * 1e4 / 344), (688, 1.1 * 2e4 / 688),
         (2432, 1.1 * 172137.56 / 2432), (7296, 1.1 * 1e6 / 7296), (1, 1.1), (3, 110.0)]


@pytest.mark.parametrize("size", SIZES, ids=lambda s: "B%d" % s[0])
@pytest.mark.parametrize("n,nw", [(1, 1), (2, 2432), (700, 1216), (1600, 3040), (2432, 2432),
                                  (3000, 3648), (4096, 4096), (5000, 5000)])
def test_equal_runs_are_covered(lib, size, n, nw):
    B, fill = [size[0]] * n, [size[1]] * n
    _check(_cuts(lib, B, fill, nw), B)


@pytest.mark.parametrize("seed", range(20))
def test_uneven_runs_are_covered(lib, seed):
    rng = np.random.default_rng(seed)
    n = int(np.exp(rng.uniform(0.0, np.log(5000.0))))
    i = rng.integers(0, len(SIZES), n)
    B, fill = [SIZES[k][0] for k in i], [SIZES[k][1] for k in i]
    for nw in (n, n + 1, 2 * n - 1, 2432 + n):
        _check(_cuts(lib, B, fill, nw), B)


def test_fewer_warps_than_runs_is_refused(lib):
    assert _cuts(lib, [4, 4, 4], [32.0] * 3, 2) is None
