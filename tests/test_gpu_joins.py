"""Replicas and spectral states whose runs have unequal numbers of segments
(targets within one size class), against the oracle (needs a GB300): FP64 to
1e-12, integer walkers exactly, FP32 to 1e-5, as for equal ones."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import assert_same_vector, fq, pair

pytestmark = pytest.mark.gpu

TARGETS = [1.3e4, 1.9e4, 1e4]  # 445, 650 and 344 segments


def _runs(h, m, targets, mode, dt, starts):
    g, o = [], []
    for i, t in enumerate(targets):
        p = dict(mode=mode, dt=dt, target=t, seed=9, run_id=i)
        keys, amps = starts[i]
        r, c = fq().Run(h, fq().default_params(**p)), O.Run(m, O.default_params(**p))
        r.seed(fq().keys_from_ints(keys), amps, m.diagonal(m.start()), 0)
        c.seed(keys, amps, m.diagonal(m.start()), 0)
        g.append(r)
        o.append(c)
    return g, o


@pytest.mark.parametrize("mode,rtol", [(1, 1e-12), (0, 1e-12), (2, 1e-5)],
                         ids=["REAL64", "INT", "REAL32"])
@pytest.mark.parametrize("model,ds", [((O.REAL_1D, 12, 1, 12, 1.0, 4.0), [0, 3]),
                                      ((O.REAL_1D, 33, 1, 33, 1.0, 20.0), [0, 16]),
                                      ((O.REAL_2D, 4, 3, 9, 1.0, 3.0), [])],
                         ids=["real1d", "real1d-128bit", "real2d"])
def test_overlaps_of_unequal_runs_match_oracle(model, ds, mode, rtol):
    h, m = pair(*model)
    dt = 1e-3
    g, o = _runs(h, m, TARGETS, mode, dt, [([m.start()], [3000.0])] * 3)
    b = fq().Batch(g)
    b.set_overlaps(ds)
    pairs = [(0, 1), (0, 2), (1, 2)]
    for block in range(2):
        b.step(8)
        for c in o:
            c.step(8)
        rows = b.overlaps()
        for r, c in zip(g, o):
            assert_same_vector(r.export(), c.export(), rtol=rtol if mode else 0.0)
        want = np.concatenate([O.overlap(o[a], o[c], ds) for a, c in pairs])
        assert rows.shape == (8, 1 + len(want))
        assert np.allclose(rows[-1, 1:], want, rtol=rtol, atol=0), (block, rows[-1, 1:], want)
    b.close()


@pytest.mark.parametrize("mode", ["REAL64", "REAL32"])
@pytest.mark.parametrize("model", [(O.REAL_1D, 10, 1, 10, 1.0, 4.0), (O.REAL_1D, 33, 1, 33, 1.0, 20.0)],
                         ids=["64bit", "128bit"])
@pytest.mark.parametrize("order", [(0, 1, 2), (2, 0, 1), (1, 2, 0)], ids=str)
def test_spectral_states_of_unequal_runs_match_oracle(order, model, mode):
    h, m = pair(*model)
    # the states share their addresses, with amplitudes of one size, so that the
    # subtraction loses no digits beyond the tolerance; few values in FP32, where
    # a rounding changes a compression with a chance of about 1e-6 a value
    rng = np.random.default_rng(31)
    occ = W.random_occupations(m.kind, m.Lx, m.Ly, m.N, 1500 if mode == "REAL64" else 300, rng)
    keys = [m.encode(x) for x in occ]
    starts = [(keys, rng.integers(8, 80, len(keys)) * rng.choice([-0.125, 0.125], len(keys)))
              for _ in range(3)]
    targets = [TARGETS[i] for i in order]
    g, o = _runs(h, m, targets, {"REAL64": 1, "REAL32": 2}[mode], 1e-3, starts)
    tol = 1e-12 if mode == "REAL64" else 1e-5
    b = fq().Batch(g)
    b.set_spectral(3)
    for block in range(2):
        b.step(4)
        assert O.spectral_step(o, 4) == 0
        for r, c in zip(g, o):
            assert_same_vector(r.export(), c.export(), rtol=tol)
    for r, c in zip(g, o):
        gh, oh = r.history(), c.history()
        assert np.array_equal(gh["len"], oh["len"])
        for f in ("shift", "norm"):
            assert np.allclose(gh[f], oh[f], rtol=tol, atol=tol), f
    b.close()


def test_runs_of_another_size_class_are_refused():
    h = fq().Hamiltonian(1, 12, 1, 12, 1.0, 4.0)
    runs = []
    for i, t in enumerate([1e4, 2.1e4]):  # 65 and 136 full buckets
        r = fq().Run(h, fq().default_params(target=t, run_id=i))
        r.seed_default(10.0)
        runs.append(r)
    b = fq().Batch(runs)
    for call in (lambda: b.set_overlaps([]), lambda: b.set_spectral(2)):
        with pytest.raises(fq().FqError):
            call()
    b.close()


@pytest.mark.parametrize("mode,rtol", [(1, 1e-12), (0, 1e-12), (2, 1e-5)],
                         ids=["REAL64", "INT", "REAL32"])
def test_warps_that_cross_pairs_match_oracle(mode, rtol):
    """Eight replicas of 344 segments: 9632 items of 28 pairs, more than the
    join's warps, so that some begin one pair's sums after another's."""
    h, m = pair(O.REAL_1D, 12, 1, 12, 1.0, 4.0)
    g, o = _runs(h, m, [1e4] * 8, mode, 1e-3, [([m.start()], [1000.0])] * 8)
    b = fq().Batch(g)
    b.set_overlaps([0, 1, 6])
    b.step(12)
    for c in o:
        c.step(12)
    rows = b.overlaps()
    want = np.concatenate([O.overlap(o[a], o[c], [0, 1, 6]) for a in range(8) for c in range(a + 1, 8)])
    assert np.allclose(rows[-1, 1:], want, rtol=rtol, atol=0)
    b.close()
