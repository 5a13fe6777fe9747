"""The training pass of the learned Poisson start at the edges of its
kernels: channel counts below, at and above 4, 8 and 16, rows of less than a
warp, a warp, and a warp and one cell, row counts that leave warps without a
row or with an odd one.  Against central differences of the FP64 network,
within the bounds of the other gradient test."""

import numpy as np
import pytest

from oracle import nn_oracle
from paper_1507_04891_gb300 import lbm, workloads as WL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,hidden", [((3, 3, 3), 1), ((3, 9, 33), 4), ((4, 17, 31), 5),
                                          ((3, 8, 32), 8), ((3, 3, 64), 9), ((4, 18, 65), 16)])
def test_gradient(shape, hidden):
    nz, ny, nx = shape
    lat = lbm.Lattice(nx, ny, nz, 1, bjerrum=0.7, poisson="mg")
    solid, sigma = WL.random_solid(shape, seed=5, fraction=0.15)
    lat.set_walls(solid, sigma)
    fluid = ~solid
    lat.nn_init(hidden=hidden, seed=11)
    g = np.random.Generator(np.random.PCG64(12))
    params = g.uniform(-0.4, 0.4, size=lat.nn_params().size).astype(np.float32)
    lat.nn_params(params)
    x0 = np.where(fluid, g.standard_normal(shape), 0.0).astype(np.float32)
    loss, grad = lat.nn_loss_grad(x0)
    p64 = params.astype(np.float64)
    ref = nn_oracle.loss(p64, x0.astype(np.float64), fluid, hidden)
    assert abs(loss - ref) <= 1e-5 * ref
    h = 1e-5
    for k in g.choice(p64.size, size=30, replace=False):
        pp, pm = p64.copy(), p64.copy()
        pp[k] += h
        pm[k] -= h
        fd = (nn_oracle.loss(pp, x0, fluid, hidden) - nn_oracle.loss(pm, x0, fluid, hidden)) / (2 * h)
        assert abs(grad[k] - fd) <= 1e-3 * np.abs(grad).max() + 1e-4 * abs(fd), (k, grad[k], fd)
