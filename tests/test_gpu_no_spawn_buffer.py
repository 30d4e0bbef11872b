"""A run whose spawn buffers could not be allocated again after a failed growth
launches nothing: every call that would step it reports FQ_ERR_NOMEM (needs a
GB300).  The failure is made on the host, by the allocator."""
import pytest

from gpu_helpers import fq

pytestmark = pytest.mark.gpu


def test_calls_that_step_report_the_missing_buffers(monkeypatch):
    import paper_2601_19505_gb300.fciqmc as F
    full = [False]
    alloc = F._TorchAllocator.alloc
    monkeypatch.setattr(F._TorchAllocator, "alloc",
                        lambda self, ctx, n, s: None if full[0] else alloc(self, ctx, n, s))
    h = fq().Hamiltonian(1, 10, 1, 10, 1.0, 3.0)
    r = fq().Run(h, fq().default_params(target=1e3))
    r.seed_default(10.0)
    r.step(3)
    b = fq().Batch([r])
    full[0] = True
    for call in (lambda: r.reserve(0, 10 ** 6), lambda: r.step(1), lambda: r.autotune(1),
                 lambda: r.profile(1), lambda: b.step(1), lambda: b.autotune(1)):
        with pytest.raises(fq().FqError) as e:
            call()
        assert e.value.code == -2
    assert r.sync() == -2
    b.close()
    r.close()
