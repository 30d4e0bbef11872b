"""The launch shapes that a run steps with untuned, on both sides of the bucket
counts at which they change in momentum space (multiples of 3 buckets a warp)
and for 128-bit addresses (20 buckets a warp), against the oracle (needs a
GB300)."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import assert_same_vector, fq, pair, runs, seeded_vector

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,target,wpb", [
    ((O.MOM_1D, 8, 1, 8, 1.0, 4.0), 3e5, (8, 8)), ((O.MOM_1D, 8, 1, 8, 1.0, 4.0), 1e6, (4, 8)),
    ((O.MOM_1D, 8, 1, 8, 1.0, 4.0), 1.4e6, (8, 8)), ((O.MOM_1D, 32, 1, 32, 1.0, 4.0), 2.2e6, (4, 8)),
    ((O.MOM_1D, 32, 1, 32, 1.0, 4.0), 3e6, (8, 8)), ((O.REAL_2D, 8, 8, 64, 1.0, 8.0), 6.2e6, (8, 8)),
    ((O.REAL_1D, 40, 1, 40, 1.0, 8.0), 7.6e6, (4, 8))], ids=str)
def test_default_shapes_match_oracle(model, target, wpb):
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
