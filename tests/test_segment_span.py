"""Which segments of a run can hold the addresses of a segment of another
(csrc/fq_shared.h, compiled for the host): the joins of replicas and spectral
states of unequal segment counts rely on it."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2601_19505_gb300", "csrc")
WRAP = """
#include "fq_shared.h"
extern "C" void spans(unsigned n, const unsigned* seg, unsigned here, unsigned there, unsigned* lo, unsigned* hi) {
    for (unsigned i = 0; i < n; ++i) fq::segment_span(seg[i], here, there, lo[i], hi[i]);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("span")
    (d / "wrap.cpp").write_text(WRAP)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "wrap.cpp"),
                    "-o", str(d / "libspan.so")], check=True)
    return ctypes.CDLL(str(d / "libspan.so"))


@pytest.mark.parametrize("here,there", [(1, 1), (1, 7), (7, 1), (344, 361), (361, 344), (65, 21),
                                        (7296, 9728), (9728, 7296), (1 << 20, 646912), (512, 512),
                                        (268002432, 268000000), (3, 268002432)])
def test_spans_hold_every_address_and_no_more(lib, here, there):
    rng = np.random.default_rng(here + there)
    seg = np.unique(np.concatenate([np.arange(min(here, 2000)), here - 1 - np.arange(min(here, 2000)),
                                    rng.integers(0, here, 2000)])).astype(np.uint32)
    lo, hi = np.zeros_like(seg), np.zeros_like(seg)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.spans(len(seg), p(seg), here, there, p(lo), p(hi))
    # the segment of a hash h among B is floor(h B / 2^32): first and last h of each
    s = [int(x) for x in seg]
    first = [-((-x << 32) // here) for x in s]
    last = [-((-(x + 1) << 32) // here) - 1 for x in s]
    for x, f, g, a, b in zip(s, first, last, lo, hi):
        assert (f * here) >> 32 == x == (g * here) >> 32
        assert f == 0 or ((f - 1) * here) >> 32 == x - 1
        assert (a, b) == ((f * there) >> 32, (g * there) >> 32)
        assert 0 <= a <= b < there
