"""Runs of small buckets that join a batch large enough to group them, after
steps alone: they follow the oracle before, in the batch and alone again (needs
a GB300)."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import assert_same_vector, fq, pair, runs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 1, 2], ids=["INT", "REAL64", "REAL32"])
@pytest.mark.parametrize("model", [(O.REAL_1D, 12, 1, 12, 1.0, 4.0), (O.REAL_1D, 34, 1, 34, 1.0, 20.0),
                                   (O.MOM_1D, 10, 1, 10, 1.0, 0.5)], ids=["64bit", "128bit", "momentum"])
def test_grouped_runs_follow_the_oracle(model, mode):
    h, m = pair(*model)
    tol = {0: 0.0, 1: 1e-12, 2: 1e-5}[mode]
    g, o = [], []
    s = m.start()
    for i in range(40):
        a, c = runs(h, m, mode=mode, dt=1e-3, target=1e4 if i % 2 else 3e4, seed=6, run_id=i)
        a.seed_default(2000.0)
        g.append(a)
        if i in (0, 17, 38, 39):
            c.seed([s], [2000.0], m.diagonal(s), 0)
            c.set_reference([s], [2000.0])
            o.append((i, c))
    for a in g:
        a.step(3)
    before = [a.capacity() for a in g]
    b = fq().Batch(g)
    after = [a.capacity() for a in g]
    assert all(x != y for x, y in zip(before, after))  # 344 segments are 86 now
    b.step(5)
    b.sync()
    for i, c in o:
        c.step(8)
        _same(g[i], c, tol)
        assert len(g[i].sample(10 ** 6)[1]) == len(c.export()[1])
    # alone again, with larger buffers
    for i, c in o:
        g[i].reserve(2 * after[i][0], 2 * after[i][1])
        assert all(x > y for x, y in zip(g[i].capacity(), after[i]))
        g[i].step(4)
        c.step(4)
        _same(g[i], c, tol)
    # and seeded anew in the batch
    i, c = o[1]
    g[i].seed_default(500.0)
    c.seed([s], [500.0], m.diagonal(s), 0)
    c.set_reference([s], [500.0])
    b.step(3)
    b.sync()
    c.step(3)
    _same(g[i], c, tol, clear=False)
    b.close()


def _same(g, o, tol, clear=True):
    assert_same_vector(g.export(), o.export(), rtol=tol)
    k, a = g.export()
    assert np.array_equal(g.lookup(k), a)
    x, y = g.history(), o.history()
    y = y[-len(x):]
    for f in ("step", "len", "exact_steps", "inexact_steps", "n_spawns"):
        assert np.array_equal(x[f], y[f]), f
    # FP32 norms differ by their rounding, and the shift by 80 (zeta / dt) times
    # that in every step
    for f in ("norm", "hproj", "vproj") + (("shift",) if tol < 1e-5 else ()):
        assert np.allclose(x[f], y[f], rtol=max(tol, 1e-12), atol=max(tol, 1e-12) * np.max(np.abs(y[f]))), f
