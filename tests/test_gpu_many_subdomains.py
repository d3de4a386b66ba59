"""Batches of more subdomains than a grid's second dimension holds subdomain-product pairs:
the reduction of the tensor-core products (up to eight products a subdomain) takes as many
subdomains as every other kernel of the step.

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


@pytest.mark.parametrize("split,problems", [("eigen", 700), ("flux", 700), ("flux", 520)])
@pytest.mark.parametrize("use_graph", [False, True])
def test_batch_of_small_problems(B, split, problems, use_graph):
    """11200 subdomains (6 x 11200 = 67200 pairs, 8 x 11200 = 89600) and 8320 (66560): past
    65535 with the tensor products."""
    one = [inputs.random_small_problem(s, nx=16, ny=16, tiles_x=4, tiles_y=4, n_mu=0, n_phi=8,
                                       rank=2, r_aug_max=4, integrator="rk4").with_(kstep_split=split)
           for s in range(4)]
    refs = [dd_dlra.DDDLRA(wl).run(2).scalar_flux() for wl in one]
    s = B.Solver([one[i % 4] for i in range(problems)], products="tensor", use_graph=use_graph)
    s.step(2)
    rho = s.scalar_flux()
    for i in range(problems):
        ref = refs[i % 4]
        assert np.linalg.norm(s.instance_flux(rho, i) - ref) <= 1e-9 * np.linalg.norm(ref), i
    s.close()
