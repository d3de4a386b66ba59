"""The autotuner's process-wide cache keeps the engines apart, and what it times for an engine is
the work that the engine's choice decides."""
import pytest

from paper_2602_14854_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    from paper_2602_14854_gb300 import binding, build
    assert torch.cuda.is_available()
    build.build()
    binding.load()
    return binding


def tuned(B, wl, **kw):
    s = B.Solver(wl, autotune=True, **kw)
    out = s.r_cap, *s.tuning()
    s.close()
    return out


def test_each_engine_has_its_own_trial(B):
    """At one even capacity (12) the two forced engines have the same shape; each gets its own
    timings, and a second solver of either the cached ones."""
    wl = inputs.random_small_problem(6, nx=36, ny=36, n_mu=4, n_phi=19, rank=4, r_aug_max=12)
    a, b = tuned(B, wl, products="fp64"), tuned(B, wl, products="tensor")
    assert a[0] == b[0] == 12
    assert (a[2][2], a[2][6]) != (b[2][2], b[2][6])
    assert tuned(B, wl, products="fp64") == a and tuned(B, wl, products="tensor") == b
