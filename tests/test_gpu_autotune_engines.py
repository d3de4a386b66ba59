"""The autotuner's process-wide cache keeps the engines apart; the engine that products = auto takes
without tuning follows the rows that subdomains have, not the tiles that they would pad."""
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


@pytest.mark.parametrize("cells,directions,rank,engine", [(4, 8, 2, 0), (10, 96, 4, 0), (11, 127, 4, 0),
                                                          (10, 96, 20, 1), (12, 128, 4, 1)])
def test_untuned_rule_for_subdomains_below_a_tile(B, cells, directions, rank, engine):
    """400 subdomains of cells x cells: the tensor cores where a subdomain fills a 128-row tile or the
    work is enough for them; subdomains of a few rows stay on the FP64 kernels, many as they
    are."""
    wl = inputs.random_small_problem(3, nx=20 * cells, ny=20 * cells, tiles_x=20, tiles_y=20, n_mu=0,
                                     n_phi=directions, rank=rank, r_aug_max=2 * rank)
    s = B.Solver(wl, products="auto")
    choice, _ = s.tuning()
    s.close()
    assert [choice[k] for k in ("oz_spatial", "oz_angular", "oz_gram_spatial", "oz_gram_angular")] == [engine] * 4
