"""Steps of neutral lattices whose launches overlap (grids of at most one
wave): two lattices stepped in turn on one caller's stream, beside each of
them alone on the library's stream, and fields read on another stream behind
an event."""

import numpy as np
import pytest

from paper_1507_04891_gb300 import lbm, workloads as WL

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def make(shape, seed, storage):
    wl = WL.binary_random(shape, seed)
    lat = lbm.Lattice(shape[2], shape[1], shape[0], 2, omega_drag=1.3, storage=storage)
    for s in range(2):
        lat.set_species(s, 1.0, 0.0, wl.n0[s], wl.u0[s])
    return lat


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("shape", [(8, 8, 16), (32, 32, 32), (40, 48, 64)])  # the last more than a wave
def test_two_lattices_in_turn(shape, storage):
    a, b = make(shape, 1, storage), make(shape, 2, storage)
    st, other = torch.cuda.Stream(), torch.cuda.Stream()
    n = torch.zeros((2,) + shape, dtype=torch.float64, device="cuda")
    for k in range(6):
        a.step(1 + k % 3, stream=st.cuda_stream)
        b.step(1 + (k + 1) % 3, stream=st.cuda_stream)
    a.get_moments_dev(0, n[0].data_ptr(), stream=st.cuda_stream)
    done = torch.cuda.Event()
    done.record(st)
    other.wait_event(done)
    b.get_moments_dev(1, n[1].data_ptr(), stream=other.cuda_stream)
    torch.cuda.synchronize()
    ra, rb = make(shape, 1, storage), make(shape, 2, storage)
    ra.step(12)
    rb.step(12)
    assert np.array_equal(n[0].cpu().numpy(), ra.get_moments(0)[0])
    assert np.array_equal(n[1].cpu().numpy(), rb.get_moments(1)[0])
    for s in range(2):
        assert np.array_equal(a.get_populations(s), ra.get_populations(s))
        assert np.array_equal(b.get_populations(s), rb.get_populations(s))
