"""A captured step whose launches the runtime refuses (more subdomains than a grid's second
dimension) is never run, and every call says so."""
import numpy as np
import pytest

from paper_2602_14854_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_a_graph_with_a_refused_launch_is_not_kept():
    import torch
    from paper_2602_14854_gb300 import binding as B, build
    assert torch.cuda.is_available()
    build.build()
    # 257 x 256 = 65792 subdomains of one cell
    wl = inputs.random_small_problem(1, nx=257, ny=256, tiles_x=257, tiles_y=256, n_mu=0, n_phi=4,
                                     rank=1, r_aug_max=2)
    s = B.Solver(wl, use_graph=True)
    before = [s.get_factors(k) for k in (0, 65791)]
    for _ in range(2):
        with pytest.raises(B.DDError):
            s.step(1)
    for (U, S, V), (U1, S1, V1) in zip(before, [s.get_factors(k) for k in (0, 65791)]):
        assert np.array_equal(U, U1) and np.array_equal(S, S1) and np.array_equal(V, V1)
    s.close()
    # the library goes on
    t = B.Solver(inputs.random_small_problem(1, nx=8, ny=8), use_graph=True)
    t.step(2)
    t.sync()
    t.close()
