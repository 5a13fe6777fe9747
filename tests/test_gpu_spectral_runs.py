"""The z solve and the source means of the spectral Poisson solver on runs of
every awkward length: one and two planes, the edges of the solve's blocks of
eight rows, runs that wrap around the periodic axis, a whole periodic axis
that is not a power of two, planes smaller than a CTA of the charge pass."""

import numpy as np
import pytest

import oracle as O
from paper_1507_04891_gb300 import lbm

pytestmark = pytest.mark.gpu


def stack(nx, ny, widths, first_wall=0):
    """Wall planes with fluid runs of the given widths between them; the last
    run wraps around when first_wall > 0."""
    nz = sum(w + 1 for w in widths)
    solid = np.zeros((nz, ny, nx), bool)
    sigma = np.zeros((nz, ny, nx))
    z = first_wall
    for k, w in enumerate(widths):
        solid[z % nz] = True
        sigma[z % nz] = -0.004 - 0.002 * k
        z += w + 1
    return solid, sigma


CASES = [(8, 8, [1, 2, 3], 0), (8, 8, [7, 8, 9], 0), (16, 8, [15, 16, 17], 0),
         (8, 16, [1, 33], 5), (32, 8, [50], 0), (16, 16, [24, 6], 9)]


@pytest.mark.parametrize("nx,ny,widths,first", CASES)
def test_solve_between_walls(nx, ny, widths, first):
    solid, sigma = stack(nx, ny, widths, first)
    g = np.random.Generator(np.random.PCG64(5))
    rho = np.where(solid, 0.0, g.uniform(-0.003, 0.003, size=solid.shape))
    lat = lbm.Lattice(nx, ny, solid.shape[0], 1, bjerrum=0.7, poisson="fft", poisson_maxit=50)
    lat.set_walls(solid, sigma)
    psi, iters, res, st = lat.solve_poisson(rho, tol=1e-10)
    assert st == lbm.LBM_OK and res <= 1e-10 and iters <= 4
    p = O.Params(1.0, 1.0, [1.0], [1.0], bjerrum=0.7, solid=solid, sigma=sigma)
    s = O.poisson_source(rho, p, solid.shape)
    so = O.PoissonSolver(~solid)
    ref = so.solve(s)[~solid]
    d = so._zero_mean(psi[~solid]) - ref
    assert np.abs(d).max() <= 1e-8 * np.abs(ref).max()


@pytest.mark.parametrize("nz", [3, 5, 9, 12, 33, 48])
def test_solve_on_a_periodic_axis(nz):
    g = np.random.Generator(np.random.PCG64(nz))
    rho = g.uniform(-0.003, 0.003, size=(nz, 8, 16))
    lat = lbm.Lattice(16, 8, nz, 1, bjerrum=0.7, poisson="fft", poisson_maxit=50)
    psi, iters, res, st = lat.solve_poisson(rho, tol=1e-10)
    assert st == lbm.LBM_OK and res <= 1e-10 and iters <= 4
    k2 = [2.0 - 2.0 * np.cos(2 * np.pi * np.arange(n) / n) for n in rho.shape]
    lam = k2[0][:, None, None] + k2[1][None, :, None] + k2[2][None, None, :]
    lam[0, 0, 0] = 1.0
    h = np.fft.fftn(4.0 * np.pi * 0.7 * rho)
    h[0, 0, 0] = 0.0
    ref = np.fft.ifftn(h / lam).real
    assert np.abs(psi - psi.mean() - ref).max() <= 1e-8 * np.abs(ref).max()


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("nx,ny,widths,first", CASES)
def test_steps_between_walls(nx, ny, widths, first, graph):
    """The charge pass's sums as source means: ten steps of a charged ternary
    mixture against the oracle, per node within the 1e-5 of the other parity
    tests."""
    solid, sigma = stack(nx, ny, widths, first)
    g = np.random.Generator(np.random.PCG64(11))
    ions = 0.01 + g.uniform(-1e-3, 1e-3, size=(2,) + solid.shape)
    n0 = np.stack([1.0 - ions[0] - ions[1], ions[0], ions[1]])
    z = np.array([0.0, 1.0, -1.0])
    lat = lbm.Lattice(nx, ny, solid.shape[0], 3, omega_drag=1.2, bjerrum=0.7,
                      e_ext=(1e-4, 0.0, 0.0), poisson="fft", step_graph=graph)
    lat.set_walls(solid, sigma)
    for s in range(3):
        lat.set_species(s, 1.0, z[s], np.where(solid, 1.0, n0[s]))
    lat.step(10)
    p = O.Params(1.0, 1.2, np.ones(3), z, bjerrum=0.7, e_ext=(1e-4, 0.0, 0.0), solid=solid,
                 sigma=sigma)
    o = O.Oracle(p, solid.shape)
    o.initialise(np.where(solid[None], 0.0, n0))
    o.run(10)
    n_o, u_o = o.fields()
    for s in range(3):
        n, u = lat.get_moments(s)
        assert (np.abs(n - n_o[s])[~solid] / n_o[s][~solid]).max() <= 1e-5
        cs = 1.0 / np.sqrt(3.0)
        assert np.abs(u - u_o[s])[:, ~solid].max() <= 1e-5 * cs
