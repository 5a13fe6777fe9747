"""Shared memory of the spectral solver's kernels: runs of 127 to 129 planes
(the z solve asks for 48 KB of dynamic memory at 128), and a plan that is used
again after a smaller one was made."""

import numpy as np
import pytest

from paper_1507_04891_gb300 import lbm

pytestmark = pytest.mark.gpu


def slit(nx, ny, width):
    solid = np.zeros((width + 2, ny, nx), bool)
    solid[0] = solid[-1] = True
    lat = lbm.Lattice(nx, ny, width + 2, 1, bjerrum=0.7, poisson="fft", poisson_maxit=50)
    lat.set_walls(solid, np.where(solid, -0.004, 0.0))
    rho = np.random.Generator(np.random.PCG64(width)).uniform(-0.003, 0.003, size=solid.shape)
    return lat, np.where(solid, 0.0, rho)


def solves(lat, rho):
    _, iters, res, st = lat.solve_poisson(rho, tol=1e-10)
    assert st == lbm.LBM_OK and res <= 1e-10 and iters <= 8


@pytest.mark.parametrize("width", [127, 128, 129, 200])
def test_long_runs(width):
    solves(*slit(8, 8, width))


def test_plans_of_several_sizes():
    a, b, c = slit(128, 128, 300), slit(128, 64, 150), slit(8, 8, 10)
    for lat, rho in (a, b, c, a):
        solves(lat, rho)
