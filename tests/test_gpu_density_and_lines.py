"""Two edges: the density of a state with empty subdomains (rank 0), at odd and even column
capacities, and the longest line that a solver accepts (side x r_aug_max = 6144), one cell past
which is refused.

Bound: 1e-9 rel-L2 on the scalar flux, the parity bound of the FP64 form."""
import numpy as np
import pytest

from oracle import dd_dlra
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


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("products,rank,cap", [("fp64", 1, 3), ("fp64", 5, 15), ("fp64", 4, 12),
                                               ("tensor", 1, 4), ("tensor", 5, 16), ("auto", 5, 16)])
def test_density_with_empty_subdomains(B, products, rank, cap):
    """The initial state, of rank 1 on one of six subdomains and 0 on the others.  (Its steps are
    ill-conditioned: noise of 1e-15 in the directions moves the oracle's own density by 1e-3.)"""
    wl = inputs.random_small_problem(3, nx=48, ny=40, xcuts=[0, 9, 41, 48], ycuts=[0, 8, 40], n_mu=3,
                                     n_phi=11, rank=rank, r_aug_max=2 * rank)
    g0 = wl.g0.reshape(40, 48).copy()
    g0[:, 9:] = 0.0
    g0[8:, :] = 0.0
    wl = wl.with_(g0=g0.reshape(-1))
    o = dd_dlra.DDDLRA(wl)
    s = B.Solver(wl, products=products)
    assert s.r_cap == cap
    assert sorted(o.ranks()) == [0] * 5 + [1] and list(s.ranks()[0]) == o.ranks()
    assert rel(s.scalar_flux(), o.scalar_flux()) <= 1e-9
    s.close()


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("split", ["eigen", "flux"])
def test_longest_line(B, axis, split):
    def problem(length):
        cuts = ([0, length], [0, 2, 5])
        xc, yc = cuts if axis == 0 else cuts[::-1]
        wl = inputs.random_small_problem(3, nx=xc[-1], ny=yc[-1], n_mu=2, n_phi=9, rank=3,
                                         r_aug_max=6, integrator="rk4", xcuts=xc, ycuts=yc)
        return wl.with_(kstep_split=split, dt=1e-4)

    wl = problem(1024)
    o = dd_dlra.DDDLRA(wl).run(2)
    s = B.Solver(wl)
    s.step(2)
    assert list(s.ranks()[0]) == o.ranks()
    assert rel(s.scalar_flux(), o.scalar_flux()) <= 1e-9
    s.close()
    with pytest.raises(B.DDError):
        B.Solver(problem(1025))
