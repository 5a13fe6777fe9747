"""The charge pass beside walls: rows of 4 to 68 nodes (quads of a row, rows
that end inside a group of 32 nodes, rows that take one node per thread),
walls that leave groups of wall nodes, of fluid nodes and of both, in every
storage format.  The first step's potential solves, under the oracle's FP64
operator, for the charge of the moments read back before the step (the same
populations, summed with compensation): the pass sums 19 values per species
in FP32 (19 x 6e-8) and two species of like size cancel, 1e-5 of the source;
a value pulled from the wrong place is a tenth of a per cent."""

import numpy as np
import pytest

import oracle as O
from paper_1507_04891_gb300 import lbm, workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("solver,walls,shape", [
    ("mg", "random", (6, 5, 4)), ("mg", "random", (5, 6, 36)), ("mg", "slab", (9, 4, 68)),
    ("mg", "random", (6, 5, 34)), ("fft", "slab", (9, 8, 8)), ("fft", "slab", (7, 16, 8)),
    ("fft", "slab", (8, 32, 32)), ("fft", "slab", (6, 64, 64))])
def test_source_of_the_first_step(solver, walls, shape, storage):
    nz, ny, nx = shape
    wl = WL.ternary_bulk(shape=shape, seed=3, spread=5e-3)
    if walls == "random":
        solid, sigma = WL.random_solid(shape, seed=4, fraction=0.1)
    else:
        solid = np.zeros(shape, bool)
        solid[2:4] = True
        sigma = np.where(solid, -0.004, 0.0)
    z = np.array([0.0, 1.0, -1.0])
    lat = lbm.Lattice(nx, ny, nz, 3, omega_drag=1.1, bjerrum=0.7, storage=storage, poisson=solver,
                      poisson_maxit=400)
    lat.set_walls(solid, sigma)
    for s in range(3):
        lat.set_species(s, 1.0, z[s], np.where(solid, 1.0, wl.n0[s]))
    n = np.stack([lat.get_moments(s)[0] for s in range(3)])
    lat.step(1)
    psi = lat.get_potential()
    p = O.Params(1.0, 1.1, np.ones(3), z, bjerrum=0.7, solid=solid, sigma=sigma)
    src = O.poisson_source(np.where(solid, 0.0, np.tensordot(z, n, 1)), p, shape)
    assert O.PoissonSolver(~solid).residual(psi, src) <= 1e-5
