"""With the FP64 products a problem's density is the same, bit for bit, alone and in a batch beside
a problem with larger subdomains: its sums are cut by its own rows."""
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


def density(B, wls):
    s = B.Solver(wls, products="fp64")
    s.step(2)
    rho = s.scalar_flux()
    out = [s.instance_flux(rho, i).copy() for i in range(len(wls))]
    s.close()
    return out


@pytest.mark.parametrize("integrator", ["euler", "rk4"])
@pytest.mark.parametrize("nx,ny", [(32, 32), (38, 26), (20, 46), (9, 7)])
def test_small_beside_large(B, nx, ny, integrator):
    kw = dict(n_mu=4, n_phi=32, rank=4, r_aug_max=8, integrator=integrator)
    small = inputs.random_small_problem(3, nx=nx, ny=ny, xcuts=[0, nx // 2, nx], ycuts=[0, ny // 2, ny],
                                        **kw)
    large = inputs.random_small_problem(5, nx=128, ny=128, **kw)        # 4 x 4096 cells
    alone = density(B, [small])[0], density(B, [large])[0]
    batch = density(B, [small, large])
    assert np.array_equal(batch[0], alone[0])
    assert np.array_equal(batch[1], alone[1])
