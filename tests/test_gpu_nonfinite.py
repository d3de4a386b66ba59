"""A NaN or an infinity in a stored factor is reported (DD_ERR_NONFINITE) after the next step, by
every form of the products: the fixed-point splitting of the tensor-core products must not turn
it into a large finite number."""
import numpy as np
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


def step_with(B, wl, factor, place, bad, **kw):
    """The error of a step from a state with one bad entry in subdomain 0's factor (None: none)."""
    s = B.Solver(wl, **kw)
    s.step(1)
    s.sync()
    f = list(s.get_factors(0))
    i = "USV".index(factor)
    f[i] = f[i].copy()
    f[i][place[0] % f[i].shape[0], place[1] % f[i].shape[1]] = bad
    s.set_factors(0, *f)
    try:
        s.step(1)
        s.scalar_flux()
        return None
    except B.DDError as e:
        return str(e)
    finally:
        s.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("factor", ["U", "S", "V"])
@pytest.mark.parametrize("products", ["fp64", "tensor"])
@pytest.mark.parametrize("precision", ["fp64", "tf32"])
def test_reported(B, products, precision, factor, bad):
    # amplitudes of 1 and 1e-6; an inner cell, the first and the last row; first and last column
    for amp in (1.0, 1e-6):
        wl = inputs.random_small_problem(3, nx=24, ny=24, n_mu=4, n_phi=16, rank=4, r_aug_max=8,
                                         integrator="rk4")
        wl = wl.with_(g0=amp * wl.g0, source=amp * wl.source)
        for place in ((70, 3), (0, 0), (-1, -1)):
            e = step_with(B, wl, factor, place, bad, products=products, precision=precision)
            assert e is not None and "NONFINITE" in e, (amp, place, e)


@pytest.mark.parametrize("rank", [4, 16, 17, 21])
@pytest.mark.parametrize("integrator", ["euler", "rk4"])
def test_reported_at_every_padded_width(B, rank, integrator):
    """Inner dimensions of 16 to 64 columns, two stages of digit planes and one."""
    wl = inputs.random_small_problem(5, nx=30, ny=26, n_mu=4, n_phi=19, rank=rank,
                                     r_aug_max=min(2 * rank, 42), integrator=integrator)
    for column in (0, rank - 1):
        e = step_with(B, wl, "U", (130, column), float("nan"), products="tensor")
        assert e is not None and "NONFINITE" in e, (column, e)
