"""The tail rule of Algorithms 4 and 5 on the GPU against the oracle's over tolerances of every
size and sign, ranks up to the column capacity: r is the smallest rank whose tail
(sum_{j >= r} sigma_j^2)^(1/2) is within the tolerance; a tolerance below zero cuts nothing.

Bound: the stored ranks exactly, the scalar flux to 1e-9 (the FP64 form's
parity bound)."""
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


@pytest.mark.parametrize("tol", [-1.0, -1e-2, -1e-300, 0.0, 1e-300, 1e-170, 2e-3, 3e-2, 10.0, 1e200])
@pytest.mark.parametrize("rank", [4, 21])
def test_ranks(B, tol, rank):
    wl = inputs.random_small_problem(3, nx=20, ny=18, n_mu=4, n_phi=19, rank=rank,
                                     r_aug_max=2 * rank)
    wl = wl.with_(rank_mode="tol", tol=tol, r_min=1, r_max=rank)
    ref = dd_dlra.DDDLRA(wl).run(2)
    s = B.Solver(wl)
    s.step(2)
    rho, ranks = s.scalar_flux(), list(s.ranks()[0])
    s.close()
    assert ranks == ref.ranks()
    r = ref.scalar_flux()
    assert np.linalg.norm(rho - r) <= 1e-9 * np.linalg.norm(r)
