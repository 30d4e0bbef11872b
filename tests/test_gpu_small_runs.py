"""Runs with fewer segments than a block has warps (needs a GB300): the warps
without a segment add nothing, so every row and the vector follow the oracle."""
import numpy as np
import pytest

from gpu_helpers import assert_same_vector, pair, runs
from test_gpu_parity import MODELS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["REAL64", "INT"])
@pytest.mark.parametrize("target", [100.0, 300.0, 600.0, 2500.0])
@pytest.mark.parametrize("model", [MODELS[0], MODELS[2]], ids=["real1d", "real2d"])
def test_few_segments_match_oracle(model, target, mode):
    h, m = pair(*model)
    g, o = runs(h, m, mode={"REAL64": 1, "INT": 0}[mode], dt=0.005, target=target, seed=4)
    weight = float(int(target / 4))
    g.seed_default(weight)
    s = m.start()
    o.seed([s], [weight], m.diagonal(s), 0)
    o.set_reference([s], [weight])
    g.step(40)
    o.step(40)
    gh, oh = g.history(), o.history()
    for f in ("step", "len", "exact_steps", "inexact_steps", "n_spawns"):
        assert np.array_equal(gh[f], oh[f]), f
    assert_same_vector(g.export(), o.export(), rtol=1e-12 if mode == "REAL64" else 0.0)
    g.close()
