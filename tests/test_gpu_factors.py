"""Diagonal factors over the whole range of sum n(n-1) / 2, condensates in real
space included, follow the oracle (needs a GB300)."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import assert_same_vector, fq, pair, runs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["REAL64", "REAL32", "INT"])
@pytest.mark.parametrize("model", [(O.REAL_1D, 8, 1, 40, 1.0, 0.05), (O.REAL_2D, 8, 8, 64, 1.0, 0.02)],
                         ids=["64bit", "128bit"])
def test_condensed_addresses_match_oracle(model, mode):
    h, m = pair(*model)
    N, M = model[3], model[1] * model[2]
    occs = []
    for top in (N, N - 1, 24, 23, 22, 5):
        occ = np.zeros(M, dtype=np.uint8)
        occ[0] = top
        occ[1] += (N - top) // 2
        occ[2] += N - top - (N - top) // 2
        occs.append(occ)
    keys = [m.encode(o) for o in occs]
    amps = [40.0, -30.0, 50.0, 60.0, 70.0, 80.0]
    g, o = runs(h, m, mode={"REAL64": 1, "REAL32": 2, "INT": 0}[mode], dt=0.001, target=1000.0,
                seed=5, capacity_vec=20000, capacity_spawn=200000)
    g.seed(fq().keys_from_ints(keys), amps, 3.0, step=7)
    o.seed(keys, amps, 3.0, step=7)
    for _ in range(3):
        g.step(1)
        o.step(1)
        assert_same_vector(g.export(), o.export(),
                           rtol={"REAL64": 1e-12, "REAL32": 1e-5, "INT": 0.0}[mode])
    tol = 1e-12 if mode != "REAL32" else 1e-5
    assert np.allclose(g.history()["shift"], o.history()["shift"], rtol=tol, atol=tol)
