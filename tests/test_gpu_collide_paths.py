"""The stream/collide's load paths at their edges: rows of 2 to 66 nodes (one
pair, rows that end inside a warp, odd rows, which take one node per thread),
node counts that are no multiple of 32, walls that leave warps of wall nodes,
of fluid nodes and of both, in every storage format, against the oracle per
node within the bounds of the other parity tests (1e-5 in FP32, 1e-3 in the
FP16, 1e-2 in BF16 with its eight mantissa bits; both round stochastically)."""

import numpy as np
import pytest

import oracle as O
from paper_1507_04891_gb300 import lbm, workloads as WL

pytestmark = pytest.mark.gpu

BOUND = {"fp32": 1e-5, "fp16": 1e-3, "bf16": 1e-2}


def case(shape, walls, seed):
    wl = WL.ternary_bulk(shape=shape, seed=seed, spread=2e-3)
    if walls == "none":
        return wl.n0, None, None
    if walls == "random":
        solid, sigma = WL.random_solid(shape, seed=seed + 1, fraction=0.12)
    else:  # a slab: whole warps of wall nodes, rows beside it, clear rows
        solid = np.zeros(shape, bool)
        solid[2:4] = True
        sigma = np.where(solid, -0.004, 0.0)
    n0 = np.where(solid[None], 1.0, wl.n0)
    return n0, solid, sigma


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("walls", ["none", "random", "slab"])
@pytest.mark.parametrize("shape", [(7, 5, 2), (8, 9, 6), (7, 6, 34), (8, 5, 66), (7, 6, 33)])
def test_steps_against_oracle(shape, walls, storage):
    n0, solid, sigma = case(shape, walls, 17)
    nz, ny, nx = shape
    z = np.array([0.0, 1.0, -1.0])
    lat = lbm.Lattice(nx, ny, nz, 3, omega_drag=1.1, bjerrum=0.7, e_ext=(1e-4, 0.0, 0.0),
                      storage=storage, poisson="mg", poisson_maxit=400)
    if solid is not None:
        lat.set_walls(solid, sigma)
    for s in range(3):
        lat.set_species(s, 1.0, z[s], n0[s])
    lat.step(8)
    p = O.Params(1.0, 1.1, np.ones(3), z, bjerrum=0.7, e_ext=(1e-4, 0.0, 0.0), solid=solid,
                 sigma=sigma)
    o = O.Oracle(p, shape)
    o.initialise(n0 if solid is None else np.where(solid[None], 0.0, n0))
    o.run(8)
    n_o, u_o = o.fields()
    fl = np.ones(shape, bool) if solid is None else ~solid
    cs = 1.0 / np.sqrt(3.0)
    for s in range(3):
        n, u = lat.get_moments(s)
        assert (np.abs(n - n_o[s])[fl] / n_o[s][fl]).max() <= BOUND[storage]
        assert np.abs(u - u_o[s])[:, fl].max() <= BOUND[storage] * cs
    # the last step's diagnostics sum the state it stored: two nodes of a
    # thread, masked wall nodes, the last warp's missing nodes
    d = lat.diagnostics()
    mass = np.array([lat.get_moments(s)[0][fl].sum() for s in range(3)])
    assert np.abs(d["mass"] - mass).max() <= 1e-6 * mass.max()

