"""The precision of a step from states met part of the way through a run: the distance of the
density from the oracle's, which is of the size of FP64 rounding there.

Bound: the geometric mean over 64 states is at most 1.2 times 4.02e-15, what the step gave with
rounded double-float pairs as the operands of the small factorisations and an FP64 refinement of
the Gram's eigenvectors (the mean's own uncertainty is 5%).  With operands truncated to 24 + 24
bits it is 5.9e-15."""
import numpy as np
import pytest

from oracle import dd_dlra
from paper_2602_14854_gb300 import inputs

pytestmark = pytest.mark.gpu


def smooth_problem(seed):
    """A Gaussian of width 0.1 near the middle, random materials, 2 x 2 uneven subdomains."""
    nx, ny = 31, 29
    wl = inputs.random_small_problem(300 + seed, nx=nx, ny=ny, xcuts=[0, 14, 31], ycuts=[0, 15, 29],
                                     n_mu=0, n_phi=45, rank=5, r_aug_max=10, integrator="rk4")
    X, Y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / nx)
    cx, cy = np.random.default_rng(seed).uniform(0.4, 0.6, 2)
    g0 = np.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / (2 * 0.1 ** 2)).reshape(-1)
    return wl.with_(g0=g0, source=np.zeros(nx * ny))


def test_error_of_a_step():
    import torch
    from paper_2602_14854_gb300 import binding as B, build
    assert torch.cuda.is_available()
    build.build()
    logs = []
    for seed in range(64):
        wl = smooth_problem(seed)
        o = dd_dlra.DDDLRA(wl).run(12)
        s = B.Solver(wl)
        for k, f in enumerate(o.state):
            s.set_factors(k, *f)
        ref = o.run(1).scalar_flux()
        s.step(1)
        rho = s.scalar_flux()
        s.close()
        logs.append(np.log(np.linalg.norm(rho - ref) / np.linalg.norm(ref)))
    assert np.exp(np.mean(logs)) <= 1.2 * 4.02e-15
