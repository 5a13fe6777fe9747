"""What setting up a lattice copies and clears is in place before its kernels
run: lattices made alike, used at once, give the same fields bit for bit.
(The face mask of the multigrid was cleared in another stream than the kernel
that fills it; cleared late, it closed every face and the solve ended at
once.)"""

import numpy as np
import pytest

from paper_1507_04891_gb300 import lbm, workloads as WL

pytestmark = pytest.mark.gpu


def make(shape, solver):
    g = np.random.Generator(np.random.PCG64(12))
    nz, ny, nx = shape
    if solver == "fft":
        solid = np.zeros(shape, bool)
        solid[0] = solid[-1] = True
        sigma = np.where(solid, -0.004, 0.0)
    else:
        solid, sigma = WL.random_solid(shape, seed=5, fraction=0.12)
    base = np.array([0.8, 0.06, 0.05])
    n0 = base[:, None, None, None] * (1.0 + g.uniform(-0.2, 0.2, size=(3,) + shape))
    lat = lbm.Lattice(nx, ny, nz, 3, omega_drag=1.1, bjerrum=0.7, poisson=solver, poisson_maxit=400)
    lat.set_walls(solid, sigma)
    for s, z in enumerate((0.0, 1.0, -1.0)):
        lat.set_species(s, 1.0, z, np.where(solid, 1.0, n0[s]))
    lat.set_plane_omega_drag(np.linspace(0.8, 1.2, nz))
    lat.step(1)
    return lat


@pytest.mark.parametrize("shape,solver", [((8, 5, 66), "mg"), ((7, 6, 34), "mg"), ((16, 16, 16), "mg"),
                                          ((33, 40, 48), "mg"), ((12, 8, 32), "fft")])
def test_lattices_made_alike_agree(shape, solver):
    seen = set()
    for _ in range(25):
        lat = make(shape, solver)
        assert lat.diagnostics()["poisson_iters"] > 0
        seen.add((lat.get_potential().tobytes(), lat.get_populations(1).tobytes()))
        lat.destroy()
    assert len(seen) == 1
