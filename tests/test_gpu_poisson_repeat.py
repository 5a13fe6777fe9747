"""Multigrid and SOR solves around odd periodic extents repeat bit for bit:
the first and the last cell of such an axis have one colour, and their
updates must not depend on which comes first.  Extents odd on the finest
level, on levels of grid kernels, on levels in shared memory, on one axis
only; a fixed number of cycles, so that the sums of the convergence test,
whose order is free, play no part."""

import numpy as np
import pytest

from paper_1507_04891_gb300 import lbm, workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("solver,shape,maxit", [
    ("mg", (75, 50, 90), 5),    # 45x25x38 and 23x13x19 by grid kernels, 12x7x10 in shared memory
    ("mg", (50, 50, 100), 5),   # even, then 25 and 13 cells
    ("mg", (33, 18, 21), 5), ("mg", (16, 27, 16), 5), ("mg", (5, 7, 9), 4), ("mg", (3, 5, 40), 4),
    ("sor", (9, 10, 11), 20), ("sor", (16, 16, 33), 20), ("sor", (27, 32, 16), 20)])
def test_same_bits_every_time(solver, shape, maxit, walls):
    nz, ny, nx = shape
    g = np.random.Generator(np.random.PCG64(3))
    rho = g.uniform(-0.01, 0.01, size=shape)
    psi0 = g.uniform(-0.01, 0.01, size=shape)
    lat = lbm.Lattice(nx, ny, nz, 1, bjerrum=0.7, poisson=solver, poisson_maxit=200)
    if walls:
        lat.set_walls(*WL.random_solid(shape, seed=9, fraction=0.1))
    runs = [lat.solve_poisson(rho, psi0=psi0, tol=1e-30, maxit=maxit) for _ in range(4)]
    assert all(r[1] == maxit and r[3] == lbm.LBM_ENOCONV for r in runs)
    assert all(np.array_equal(r[0], runs[0][0]) for r in runs[1:])
