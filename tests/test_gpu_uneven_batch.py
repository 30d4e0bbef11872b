"""Batches whose runs have segments of unequal fill: every run's rows and vector
are those of the run alone, for every walker type, address width, model and
annihilation arm (needs a GB300).  Integer walkers exactly; real ones to the
rounding of their sums (FP64 1e-12, FP32 1e-5), with equal counts."""
import numpy as np
import pytest

from gpu_helpers import assert_same_vector, fq

pytestmark = pytest.mark.gpu

TARGETS = [2e5, 300.0, 5e3, 9e4, 700.0]
SHAPES = {"ring-64bit": lambda i: (1, 8 + i, 1, 8 + i), "ring-128bit": lambda i: (1, 34 + i, 1, 34 + i),
          "lattice-128bit": lambda i: (2, 6, 6, 36 + i), "momentum": lambda i: (3, 8 + i, 1, 8 + i)}


@pytest.mark.parametrize("arm", [2, 1], ids=["hash", "sort"])
@pytest.mark.parametrize("mode", [0, 1, 2], ids=["INT", "REAL64", "REAL32"])
@pytest.mark.parametrize("shape", SHAPES)
def test_uneven_batch_rows_are_those_of_the_runs_alone(shape, mode, arm):
    def make(i):
        h = fq().Hamiltonian(*SHAPES[shape](i), 1.0, 0.5 if shape == "momentum" else 3.0)
        # the lattice grows fivefold in these steps
        r = fq().Run(h, fq().default_params(mode=mode, dt=0.001, target=TARGETS[i], seed=2, run_id=i,
                                            annihilation=arm, capacity_vec=int(20 * TARGETS[i]) + 4096,
                                            capacity_spawn=int(40 * TARGETS[i]) + 8192))
        r.seed_default(float(int(TARGETS[i] / 2)))
        return r

    tol = {0: 0.0, 1: 1e-12, 2: 1e-5}[mode]
    together = [make(i) for i in range(len(TARGETS))]
    b = fq().Batch(together)
    b.step(20)
    b.sync()
    for i, r in enumerate(together):
        a = make(i)
        a.step(20)
        x, y = r.history(), a.history()
        assert len(x) == 20
        for f in ("step", "len", "exact_steps", "inexact_steps", "n_spawns"):
            assert np.array_equal(x[f], y[f]), (i, f)
        for f in ("norm", "shift", "hproj", "vproj"):
            if mode == 0 and f != "hproj":
                assert np.array_equal(x[f], y[f]), (i, f)
            else:  # the energy's terms are added segment by segment
                rtol = max(tol, 1e-14)
                assert np.allclose(x[f], y[f], rtol=rtol, atol=rtol * np.max(np.abs(y[f]))), (i, f)
        assert_same_vector(r.export(), a.export(), rtol=tol, what="run %d" % i)
        a.close()
    b.close()
