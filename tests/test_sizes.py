"""Sizes of segments and spawn buckets (csrc/fq_sizes.h, compiled for the
host): a capacity is held, growing it grows the buckets, and the room that
small buckets have beyond it is bounded."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2601_19505_gb300", "csrc")
WRAP = """
#include "fq_sizes.h"
using namespace fq;
extern "C" unsigned segs(double s, unsigned slots, int sms) { return segments_for(s, slots, sms).B; }
extern "C" unsigned group(double s, unsigned slots, int sms) { return segments_for(s, slots, sms).group; }
extern "C" double full(double s, unsigned slots) { return full_segments(s, slots); }
extern "C" unsigned vec(double t, unsigned B) { return vec_slots(t, B); }
extern "C" unsigned spawn(unsigned B, double full, double usual, double t) {
    return spawn_room(B, full, 8.0, usual).slots(t);
}
extern "C" double total(unsigned B, double full, double usual, unsigned cs) {
    return spawn_room(B, full, 8.0, usual).total(cs);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("sizes")
    (d / "wrap.cpp").write_text(WRAP)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "wrap.cpp"),
                    "-o", str(d / "libsizes.so")], check=True)
    L = ctypes.CDLL(str(d / "libsizes.so"))
    D, U = ctypes.c_double, ctypes.c_uint
    L.full.restype = L.total.restype = D
    L.segs.restype = L.group.restype = L.vec.restype = L.spawn.restype = U
    L.group.argtypes = [D, U, ctypes.c_int]
    L.segs.argtypes, L.full.argtypes, L.vec.argtypes = [D, U, ctypes.c_int], [D, U], [D, U]
    L.spawn.argtypes, L.total.argtypes = [U, D, D, D], [U, D, D, U]
    return L


@pytest.mark.parametrize("slots", [256, 512])
@pytest.mark.parametrize("target", [10.0, 300.0, 1861.0, 1862.0, 5e3, 1e4, 7e4, 8e4, 4.2e5, 1e6, 1e8])
def test_capacities(lib, target, slots):
    s = 1.1 * target
    B, full = lib.segs(s, slots, 152), lib.full(s, slots)
    usual = 1.5 * (2.0 * target + 1024.0) + 4096.0
    assert B >= 1 and full >= 1.0
    t = 500.0
    while t <= 4e9:
        cs = lib.spawn(B, full, usual, t)
        nominal = lib.total(B, full, usual, cs)
        assert cs % 32 == 0 and cs * B >= t and nominal >= t
        # doubling what was asked for, or half as much again of what there is,
        # gives more room per bucket
        if t >= 32.0 * min(B, full):
            assert lib.spawn(B, full, usual, 2.0 * t) > cs
        assert lib.spawn(B, full, usual, 1.5 * nominal) > cs
        assert lib.spawn(B, full, usual, nominal) >= cs
        # beyond the usual sizes the buffers grow by what is asked for, up to
        # the allowance for its fluctuation
        if t > 16.0 * usual:
            most = lib.spawn(B, full, usual, 16.0 * usual)
            assert cs * B <= most * B + t + 4.0 * (8.0 * t * B) ** 0.5 + 32.0 * B
        t *= 2.0
    for t in (1e3, target, 1e8):
        assert lib.vec(t, B) * B >= t


@pytest.mark.parametrize("slots", [256, 512])
@pytest.mark.parametrize("sms", [1, 132, 152])
def test_groups_of_small_buckets_are_about_full_ones(lib, slots, sms):
    t = 10.0
    while t < 1e8:
        B, group, full = lib.segs(t, slots, sms), lib.group(t, slots, sms), lib.full(t, slots)
        warps = 16 * sms
        assert B % group == 0
        if full > warps or t < 2048.0:
            assert group == 1
        else:
            # no more buckets than warps; a group fills 1 to 3 sixths of a table
            assert B <= warps
            if group > 1:
                assert slots / 6.0 <= t * group / B <= slots / 2.0
        t *= 1.03
