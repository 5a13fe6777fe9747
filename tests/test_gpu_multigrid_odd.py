"""Multigrid on extents whose levels halve into an odd number of cells: odd
from the finest level on, odd further down, short axes, with and without
walls, a slit (not periodic along z) of odd width."""

import numpy as np
import pytest

import oracle as O
from paper_1507_04891_gb300 import lbm, workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", ["none", "random", "slit"])
@pytest.mark.parametrize("shape", [(5, 7, 9), (9, 10, 11), (17, 33, 13), (3, 5, 40), (22, 14, 38),
                                   (19, 18, 36), (33, 18, 21)])
def test_solve_against_oracle(shape, walls):
    tol = 1e-9
    nz, ny, nx = shape
    g = np.random.Generator(np.random.PCG64(7))
    solid = sigma = None
    if walls == "random":
        solid, sigma = WL.random_solid(shape, seed=9, fraction=0.1)
    elif walls == "slit":
        solid = np.zeros(shape, bool)
        solid[0] = True
        sigma = np.where(solid, -0.01, 0.0)
    rho = g.uniform(-0.01, 0.01, size=shape)
    lat = lbm.Lattice(nx, ny, nz, 1, bjerrum=0.7, poisson="mg", poisson_maxit=100)
    if solid is not None:
        lat.set_walls(solid, sigma)
    psi, iters, res, st = lat.solve_poisson(rho, tol=tol)
    assert st == lbm.LBM_OK and res <= tol and iters <= (100 if walls == "random" else 40)
    p = O.Params(1.0, 1.0, [1.0], [1.0], bjerrum=0.7, solid=solid, sigma=sigma)
    fluid = O.fluid_mask(shape, p)
    s = O.poisson_source(np.where(fluid, rho, 0.0), p, shape)
    so = O.PoissonSolver(fluid)
    assert so.residual(psi, s) <= 2 * tol
    if walls == "random":
        return
    # |e| <= |r| / lambda_min and |psi| >= |s| / 12, with the smallest
    # eigenvalue of the longest axis (a wall doubles its wavelength)
    ref = so.solve(s)[fluid]
    d = so._zero_mean(psi[fluid]) - ref
    lam = min([4 * np.sin(np.pi / n) ** 2 for n in ((ny, nx) if walls == "slit" else shape)]
              + [4 * np.sin(np.pi / (2 * (nz - 1))) ** 2])
    assert np.linalg.norm(d) <= 12 * 2 * tol / lam * np.linalg.norm(ref)
