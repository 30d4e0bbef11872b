"""Joins whose segments are too large for on-chip tables use tables in device
memory (needs a GB300): rows and states follow the oracle all the same."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_helpers import assert_same_vector, fq, pair

pytestmark = pytest.mark.gpu

# 344 segments; entries per segment, so that an overlap table is beyond 200 KB
# (16384 slots of 20 bytes, 8192 of 28) and a two-state one below 800 KB
CASES = [((O.REAL_1D, 20, 1, 20, 1.0, 2.0), 9300), ((O.REAL_1D, 33, 1, 33, 1.0, 20.0), 4000)]


def _runs(h, m, entries, n):
    rng = np.random.default_rng(5)
    keys = [m.encode(x) for x in W.random_occupations(m.kind, m.Lx, m.Ly, m.N, 1500, rng)]
    g, o = [], []
    for i in range(n):
        p = dict(mode=1, dt=1e-3, target=1e4, seed=9, run_id=i)
        amps = rng.integers(8, 80, len(keys)) * rng.choice([-0.125, 0.125], len(keys))
        r = fq().Run(h, fq().default_params(capacity_vec=344 * entries, **p))
        c = O.Run(m, O.default_params(**p))
        r.seed(fq().keys_from_ints(keys), amps, m.diagonal(m.start()), 0)
        c.seed(keys, amps, m.diagonal(m.start()), 0)
        g.append(r)
        o.append(c)
    return g, o


@pytest.mark.parametrize("model,entries", CASES, ids=["64bit", "128bit"])
def test_overlaps_of_large_segments_match_oracle(model, entries):
    h, m = pair(*model)
    g, o = _runs(h, m, entries, 3)
    b = fq().Batch(g)
    b.set_overlaps([0, 2])
    b.step(4)
    for c in o:
        c.step(4)
    want = np.concatenate([O.overlap(o[a], o[c], [0, 2]) for a, c in ((0, 1), (0, 2), (1, 2))])
    # products of both signs: their sum is right to the rounding of its terms
    size = np.concatenate([_size(o[a], o[c], m) for a, c in ((0, 1), (0, 2), (1, 2))])
    assert np.all(np.abs(b.overlaps()[-1, 1:] - want) <= 1e-12 * size)
    b.close()


def _size(a, c, m):
    """Sums of the absolute products (G2: at most N^2 / M of each)."""
    (ka, va), (kc, vc) = a.export(), c.export()
    d = dict(zip(zip(ka["lo"].tolist(), ka["hi"].tolist()), np.abs(va)))
    s = sum(d.get(k, 0.0) * v for k, v in zip(zip(kc["lo"].tolist(), kc["hi"].tolist()), np.abs(vc)))
    return [s, s * m.N ** 2 / m.M, s * m.N ** 2 / m.M]


@pytest.mark.parametrize("model,entries", CASES, ids=["64bit", "128bit"])
def test_spectral_states_of_large_segments_match_oracle(model, entries):
    h, m = pair(*model)
    g, o = _runs(h, m, entries, 2)
    b = fq().Batch(g)
    b.set_spectral(2)
    b.step(4)
    assert O.spectral_step(o, 4) == 0
    for r, c in zip(g, o):
        assert_same_vector(r.export(), c.export(), rtol=1e-12)
        assert np.array_equal(r.history()["len"], c.history()["len"])
    b.close()


def test_larger_segments_are_refused_and_the_batch_steps_on():
    h, m = pair(*CASES[0][0])
    g, o = _runs(h, m, 45000, 2)
    b = fq().Batch(g)
    for call in (lambda: b.set_overlaps([]), lambda: b.set_spectral(2)):
        with pytest.raises(fq().FqError):
            call()
    b.step(3)
    b.sync()
    for r, c in zip(g, o):
        c.step(3)
        assert_same_vector(r.export(), c.export(), rtol=1e-12)
    b.close()


def test_a_smaller_batch_leaves_an_earlier_one_its_tables():
    """Autotuning launches the join itself: it needs the on-chip memory that
    the batch was built for, whatever batches came after."""
    h, m = pair(*CASES[0][0])
    g, _ = _runs(h, m, 2000, 2)  # tables of 80 KB
    b = fq().Batch(g)
    b.set_overlaps([])
    small = [fq().Run(h, fq().default_params(target=100.0, run_id=i)) for i in range(2)]
    for r in small:
        r.seed_default(10.0)
    c = fq().Batch(small)
    c.set_overlaps([])
    b.autotune(1)
    row = b.overlaps()[-1]
    (ka, va), (kb, vb) = g[0].export(), g[1].export()
    _, ia, ib = np.intersect1d(ka["lo"], kb["lo"], return_indices=True)
    assert row[0] == g[0].stats()["step"] and len(ia) > 100
    assert abs(row[1] - np.dot(va[ia], vb[ib])) <= 1e-12 * np.dot(np.abs(va[ia]), np.abs(vb[ib]))
    b.close()
    c.close()
