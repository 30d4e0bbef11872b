"""Autotuning a batch after one of its runs has grown uses the run's new
buffers (needs a GB300): integer walkers step as the run does alone."""
import numpy as np
import pytest

from gpu_helpers import fq

pytestmark = pytest.mark.gpu


def test_batch_autotune_after_reserve():
    h = fq().Hamiltonian(1, 10, 1, 10, 1.0, 3.0)

    def make(i):
        r = fq().Run(h, fq().default_params(mode=0, dt=0.002, target=3e3, seed=4, run_id=i))
        r.seed_default(500.0)
        return r

    runs = [make(0), make(1)]
    b = fq().Batch(runs)
    b.step(4)
    runs[1].reserve(200000, 400000)
    b.autotune(1)
    n = runs[0].stats()["step"]
    assert n > 5
    b.step(3)
    b.sync()
    for i, r in enumerate(runs):
        a = make(i)
        a.step(n + 3)
        (ka, aa), (kr, ar) = a.export(), r.export()
        assert np.array_equal(ka, kr) and np.array_equal(aa, ar)
    b.close()
