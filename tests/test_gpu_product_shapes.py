"""The tensor-core product kernels, the eigenbasis K-step and the small eigen/singular value
kernels at the sizes where they can go wrong, against the FP64 oracle through the C ABI:
subdomains of one, of almost, exactly and just over a row tile (128 rows) or a read-out group
(256 rows), direction counts off every multiple, column capacities at the edges of the padded
widths (16, 32, 48, 64), one subdomain and many of very different sizes, lines cut into
segments.

Bound: 1e-9 rel-L2 on the scalar flux, the parity bound of the FP64 form (the products are
FP64-accurate: their error is a few units of 2^-54 per entry, the step's own amplification of
rounding included the other parity tests measure 1e-14 to 1e-10).
"""
import numpy as np
import pytest

from oracle import dd_dlra

pytestmark = pytest.mark.gpu

BOUND = 1e-9


@pytest.fixture(scope="module")
def B():
    import torch
    from paper_2602_14854_gb300 import binding, build
    assert torch.cuda.is_available()
    build.build()
    binding.load()
    return binding


def problem(xcuts, ycuts, n_mu, n_phi, rank, integrator="euler", seed=3, nsteps=2, **kw):
    from paper_2602_14854_gb300 import inputs
    wl = inputs.random_small_problem(seed, nx=xcuts[-1], ny=ycuts[-1], n_mu=n_mu, n_phi=n_phi,
                                     rank=rank, r_aug_max=2 * rank, integrator=integrator,
                                     xcuts=xcuts, ycuts=ycuts, nsteps=nsteps)
    return wl.with_(**kw) if kw else wl


def check(B, wl, nsteps=2, **kw):
    ref = dd_dlra.DDDLRA(wl).run(nsteps)
    s = B.Solver(wl, **kw)
    s.step(nsteps)
    rho, ranks = s.scalar_flux(), list(s.ranks()[0])
    s.close()
    r = ref.scalar_flux()
    assert ranks == ref.ranks()
    assert np.linalg.norm(rho - r) <= BOUND * np.linalg.norm(r)


# rows per subdomain: 64 .. 90 | 127, 128, 129 | 255, 256, 257 | one large among small ones
CUTS = {
    "tile": ([0, 127, 255, 384], [0, 1]),
    "group": ([0, 255, 511, 768], [0, 1]),
    "two-row": ([0, 64, 192], [0, 2, 3]),
    "uneven": ([0, 9, 41, 48], [0, 8, 40]),
    "one": ([0, 37], [0, 29]),
}


@pytest.mark.parametrize("cuts", sorted(CUTS))
@pytest.mark.parametrize("integrator", ["euler", "rk4"])
@pytest.mark.parametrize("products", ["tensor", "fp64"])
def test_rows_at_tile_edges(B, cuts, integrator, products):
    xc, yc = CUTS[cuts]
    check(B, problem(xc, yc, 3, 11, 4, integrator), products=products)


@pytest.mark.parametrize("rank", [1, 5, 6, 8, 10, 11, 16, 17, 21])
def test_column_capacities(B, rank):
    """3 r columns in the augmentation: 3, 15 | 18 (above 16) | 24, 30, 33 | 48, 51 | 63 of 64."""
    check(B, problem([0, 12, 25], [0, 11, 24], 4, 19, rank, "rk4"), products="tensor")


@pytest.mark.parametrize("n_mu,n_phi", [(0, 65), (1, 127), (3, 43), (2, 64), (5, 26), (7, 37)])
def test_direction_counts(B, n_mu, n_phi):
    """65, 127, 129, 128, 130 and 259 directions."""
    check(B, problem([0, 10, 23], [0, 13], n_mu, n_phi, 5), products="tensor")


@pytest.mark.parametrize("precision", ["mixed", "tf32", "bf16"])
def test_reduced_forms_with_the_products(B, precision):
    """The reduced forms keep their bounds with the products on the tensor cores."""
    wl = problem([0, 12, 25], [0, 11, 24], 4, 19, 6, "rk4")
    ref = dd_dlra.DDDLRA(wl).run(2).scalar_flux()
    s = B.Solver(wl, precision=precision, products="tensor")
    s.step(2)
    rho = s.scalar_flux()
    s.close()
    assert np.linalg.norm(rho - ref) <= (1e-3 if precision == "bf16" else 1e-5) * np.linalg.norm(ref)


@pytest.mark.parametrize("split", ["eigen", "flux"])
@pytest.mark.parametrize("products", ["tensor", "fp64"])
def test_inflow_on_every_side(B, split, products):
    from paper_2602_14854_gb300 import inputs
    wl = problem([0, 9, 20], [0, 8, 19], 3, 13, 4, "rk4", kstep_split=split)
    rng = np.random.default_rng(7)
    wl = wl.with_(inflow={s: (rng.uniform(0.5, 1.5, n), rng.uniform(0.0, 1.0, wl.n))
                          for s, n in (("x_lo", wl.ny), ("x_hi", wl.ny), ("y_lo", wl.nx),
                                       ("y_hi", wl.nx))})
    check(B, wl, products=products)


@pytest.mark.parametrize("length", [15, 16, 17, 32, 35, 96, 300])
@pytest.mark.parametrize("integrator", ["euler", "rk4"])
def test_line_lengths(B, length, integrator):
    """Lines shorter than a segment of the K-step, at its edges, cut into several, and longer
    than any a CTA could hold."""
    check(B, problem([0, length], [0, 3, 7], 2, 9, 3, integrator))
    check(B, problem([0, 3, 7], [0, length], 2, 9, 3, integrator))


def test_a_large_subdomain_among_small_ones(B):
    """18000 rows beside 20: more 256-row chunks than the chunk exponents have slots."""
    check(B, problem([0, 150, 154], [0, 120, 125], 2, 9, 4), products="tensor")


@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 1), (10, 2), (20, 8)])
def test_subdomain_counts(B, nx, ny):
    """1, 2, 20 and 160 subdomains: the S-step's columns over 16, 15 or fewer CTAs, down to one."""
    wl = problem(list(range(0, 4 * nx + 1, 4)), list(range(0, 3 * ny + 1, 3)), 2, 9, 3, "rk4")
    check(B, wl)
    check(B, wl, precision="fp64", products="tensor")


def test_equal_norms_take_the_sweeps(B):
    """A centred, symmetric state: singular values in exact pairs, where the simultaneous
    rotation of all pairs does not apply."""
    from paper_2602_14854_gb300 import inputs
    wl = inputs.config_c0(tiles_x=1, tiles_y=1, rank=8, nsteps=4)
    check(B, wl, nsteps=4)
    check(B, wl, nsteps=4, products="tensor")


def test_density_of_odd_shapes(B):
    """The density readout: odd and even capacities, ranks 0 .. full, uneven subdomains."""
    for rank in (1, 4, 5):
        wl = problem([0, 9, 41, 48], [0, 8, 40], 3, 11, rank)
        ref = dd_dlra.DDDLRA(wl).run(1).scalar_flux()
        s = B.Solver(wl)
        s.step(1)
        rho = s.scalar_flux()
        s.close()
        assert np.linalg.norm(rho - ref) <= BOUND * np.linalg.norm(ref)
