"""Segment counts that are no power of two, and batches whose runs have
segments of unequal fill: every run of a batch steps as it does alone, whatever
the shares of the warps (needs a GB300)."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import assert_same_vector, fq, pair, runs, seeded_vector

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("target", [1000.0, 2100.0, 5000.0, 40000.0])
@pytest.mark.parametrize("model", [(O.REAL_1D, 20, 1, 20, 1.0, 2.0), (O.REAL_2D, 8, 8, 64, 1.0, 8.0)],
                         ids=["64bit", "128bit"])
def test_segment_counts_match_oracle(model, target):
    h, m = pair(*model)
    # the lattice overshoots its target tenfold in these steps
    g, o = runs(h, m, dt=0.001, target=target, seed=3, capacity_vec=500000, capacity_spawn=2000000)
    g.seed_default(float(int(target / 2)))
    s = m.start()
    o.seed([s], [float(int(target / 2))], m.diagonal(s), 0)
    o.set_reference([s], [float(int(target / 2))])
    g.step(8)
    o.step(8)
    assert_same_vector(g.export(), o.export(), rtol=1e-12)
    k, a = g.export()
    assert np.array_equal(g.lookup(k), a)
    assert len(g.sample(10 ** 6)[1]) == len(a)
    assert np.array_equal(g.history()["n_spawns"], o.history()["n_spawns"])


@pytest.mark.parametrize("targets", [[300.0], [300.0, 2e5], [2e5, 300.0, 5e3, 9e4, 700.0],
                                     [1e3 * (1 + i) for i in range(17)]], ids=len)
def test_uneven_batch_steps_like_its_runs_alone(targets):
    def make(i, t):
        h = fq().Hamiltonian(1, 8 + i, 1, 8 + i, 1.0, 3.0)
        r = fq().Run(h, fq().default_params(mode=0, dt=0.002, target=t, seed=2, run_id=i))
        r.seed_default(float(int(t / 2)))
        return r

    together = [make(i, t) for i, t in enumerate(targets)]
    b = fq().Batch(together)
    b.step(30)
    b.sync()
    for i, t in enumerate(targets):
        r = make(i, t)
        r.step(30)
        (ka, aa), (kb, ab) = r.export(), together[i].export()
        assert np.array_equal(ka, kb) and np.array_equal(aa, ab)
        assert np.array_equal(r.history()["n_spawns"], together[i].history()["n_spawns"])
        r.close()
    b.close()


@pytest.mark.parametrize("model,target,wpb", [
    ((O.REAL_1D, 20, 1, 20, 1.0, 2.0), 8e6, (4, 4)), ((O.REAL_1D, 20, 1, 20, 1.0, 2.0), 5.5e6, (8, 8)),
    ((O.REAL_2D, 8, 8, 64, 1.0, 8.0), 8e6, (4, 8)), ((O.MOM_1D, 8, 1, 8, 1.0, 4.0), 8e5, (4, 8)),
    ((O.MOM_1D, 32, 1, 32, 1.0, 4.0), 8e6, (4, 8))], ids=str)
def test_default_shapes_match_oracle(model, target, wpb):
    """The launch shape a run steps with untuned, on both sides of the bucket
    counts at which it changes (16 buckets a warp; one in momentum space)."""
    h, m = pair(*model)
    keys, amps = seeded_vector(m, 2000, 17)
    g, o = runs(h, m, dt=0.001, target=target, seed=12)
    g.seed(fq().keys_from_ints(keys), amps, -2.0, step=5)
    o.seed(keys, amps, -2.0, step=5)
    g.step(2)
    o.step(2)
    s = g.shape()
    assert (s["spawn_wpb"], s["merge_wpb"]) == wpb
    assert_same_vector(g.export(), o.export(), rtol=1e-12)
    assert np.array_equal(g.history()["n_spawns"], o.history()["n_spawns"])
    g.close()
