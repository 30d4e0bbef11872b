"""A batch of more runs than half the resident warps: every run steps as it
does alone (needs a GB300)."""
import numpy as np
import pytest

from gpu_helpers import fq

pytestmark = pytest.mark.gpu


def test_many_equal_runs_step_alike():
    # 1900 runs of 43 segments (172 in groups of 4): more runs than half the warps of either kernel
    h = fq().Hamiltonian(1, 8, 1, 8, 1.0, 3.0)

    def make():
        r = fq().Run(h, fq().default_params(mode=0, dt=0.002, target=5e3, seed=2))
        r.seed_default(2000.0)
        return r

    alone = make()
    alone.step(6)
    rows, (ka, aa) = alone.history(), alone.export()
    together = [make() for _ in range(1900)]
    b = fq().Batch(together)
    b.step(6)
    b.sync()
    for r in together:
        h6 = r.history(cap=16)
        for f in rows.dtype.names:  # the energy's terms are added segment by segment
            assert (np.allclose(h6[f], rows[f], rtol=1e-14, atol=0) if f == "hproj"
                    else np.array_equal(h6[f], rows[f])), f
    for r in (together[0], together[950], together[-1]):
        k, a = r.export()
        assert np.array_equal(k, ka) and np.array_equal(a, aa)
    b.close()
