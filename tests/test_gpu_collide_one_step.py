"""One step of the stream/collide per population and node against an oracle
step from the same populations.

Every species starts with large differences from node to node, so that the
only thing between the two is rounding: the moving populations of the 16-bit
formats are rounded once (stochastically: less than one unit of the stored
h = f / (w n_ref) - 1), the rest population is formed from the stored moving
ones (weights over w_0: two units of theirs) and rounded once itself; FP32
arithmetic adds about sixty roundings of values below two, three times that
in the rest population.  Populations pulled from a neighbour of the right
node, or a field at rest, miss these bounds by far, which is checked too.
Rows of one pair, rows that end inside a warp, odd rows, walls that leave
warps of wall nodes, of fluid nodes and of both."""

import numpy as np
import pytest

import oracle as O
from paper_1507_04891_gb300 import lbm, workloads as WL

pytestmark = pytest.mark.gpu

Z = np.array([0.0, 1.0, -1.0])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def unit(h, storage):
    """Distance of neighbouring stored values at h."""
    if storage == "fp32":
        return np.zeros_like(h)
    e = np.floor(np.log2(np.maximum(np.abs(h), 1e-30)))
    return 2.0 ** (np.maximum(e, -14) - 10) if storage == "fp16" else 2.0 ** (e - 7)


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("walls", ["none", "random", "slab"])
@pytest.mark.parametrize("shape", [(7, 5, 2), (8, 9, 6), (7, 6, 34), (8, 5, 66), (7, 6, 33)])
def test_one_step_per_population(shape, walls, storage):
    g = np.random.Generator(np.random.PCG64(29))
    base = np.array([0.8, 0.06, 0.05])
    n0 = base[:, None, None, None] * (1.0 + g.uniform(-0.2, 0.2, size=(3,) + shape))
    u0 = g.uniform(-0.05, 0.05, size=(3, 3) + shape)
    solid = sigma = None
    if walls == "random":
        solid, sigma = WL.random_solid(shape, seed=5, fraction=0.12)
    elif walls == "slab":
        solid = np.zeros(shape, bool)
        solid[2:4] = True
        sigma = np.where(solid, -0.004, 0.0)
    fl = np.ones(shape, bool) if solid is None else ~solid
    nz, ny, nx = shape
    lat = lbm.Lattice(nx, ny, nz, 3, omega_drag=1.1, omega_visc=1.2, bjerrum=0.7,
                      e_ext=(1e-3, 0.0, -2e-3), storage=storage, poisson="mg", poisson_maxit=400)
    if solid is not None:
        lat.set_walls(solid, sigma)
    for s in range(3):
        lat.set_species(s, 1.0, Z[s], np.where(fl, n0[s], 1.0), u0[s])
    f0 = np.stack([lat.get_populations(s) for s in range(3)])
    lat.step(1)
    f1 = np.stack([lat.get_populations(s) for s in range(3)])
    o = O.Oracle(O.Params(1.2, 1.1, np.ones(3), Z, bjerrum=0.7, e_ext=(1e-3, 0.0, -2e-3),
                          solid=solid, sigma=sigma), shape)
    o.f = f0
    o.step()
    eps = 2.0 ** -24
    for s in range(3):
        wn = W[:, None] * n0[s][fl].mean()
        h, ho = f1[s][:, fl] / wn - 1.0, o.f[s][:, fl] / wn - 1.0
        u = unit(np.maximum(np.abs(h), np.abs(ho)), storage)
        bound = u + 120 * eps
        bound[0] += (W[1:, None] / W[0] * u[1:].max(axis=1, keepdims=True)).sum() + 240 * eps
        assert (np.abs(h - ho) <= bound).all(), (s, (np.abs(h - ho) / bound).max())
        # a neighbour's values, or none, are not within the bounds
        for axis in (1, 2, 3):
            other = np.roll(o.f[s], 1, axis)[:, fl] / wn - 1.0
            assert (np.abs(other - ho) > bound)[1:].mean() > 0.9
        assert (np.abs(ho) > bound)[1:].mean() > 0.9
