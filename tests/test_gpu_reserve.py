"""A run of small buckets that overflows a small spawn capacity steps on once
twice that capacity is reserved (needs a GB300)."""
import numpy as np
import pytest

from gpu_helpers import fq

pytestmark = pytest.mark.gpu


def test_reserving_twice_the_capacity_grows_the_buckets():
    # 12 sites, 344 buckets, integer walkers at the start address: every attempt
    # of the 4000 is a spawn (dt 24 sqrt(2) = 1.02) to one of 24 neighbours, all
    # in different buckets, 167 each on average (deviation 13).  3000 spawns a
    # step are 160 slots per bucket, 6000 are 224.
    h = fq().Hamiltonian(1, 12, 1, 12, 1.0, 4.0)

    def make(capacity):
        r = fq().Run(h, fq().default_params(mode=0, dt=0.03, target=1e4, seed=3,
                                            capacity_spawn=capacity))
        r.seed_default(4000.0)
        r.step(1)
        return r

    r = make(3000)
    assert r.sync() == -3 and r.error_bits() == 1
    before = r.capacity()
    r.reserve(0, 6000)
    after = r.capacity()
    assert after[0] == before[0] and after[1] > before[1] >= 3000
    r.step(1)
    assert r.sync() == 0 and r.stats()["step"] == 1
    big = make(1 << 20)
    assert big.sync() == 0
    (ka, aa), (kb, ab) = r.export(), big.export()
    assert np.array_equal(ka, kb) and np.array_equal(aa, ab)
    assert r.history().tobytes() == big.history().tobytes()
