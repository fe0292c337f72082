"""The energy sums: what they take from a state (the electrons' momenta alone for their kinetic energy), and that
they are as exact as sums in 64 bits."""
import math

import numpy as np
import pytest

from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_parity import _built, gb  # noqa: F401
from tests.test_zz_no_alloc import _view

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_electron_cells_are_not_part_of_the_kinetic_energy():
    """A state view whose electron cells were never filled in (here -1): the same five energies."""
    sim = gb().Simulation(workload("tiny", nx=48, nz=40, slab_k=20))
    sim.step(3)
    view, keep = _view(gb(), sim)
    out = torch.empty((2, 5), dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream()
    gb().pic_energy_noalloc(sim.cfg, view, out[0].data_ptr(), st.cuda_stream)
    keep[1]["cell"].fill_(-1)
    gb().pic_energy_noalloc(sim.cfg, view, out[1].data_ptr(), st.cuda_stream)
    assert out[0, 1] > 0 and torch.equal(out[0], out[1])
    sim.close()


def _terms(rng, n):
    """Momenta of one thread's particles and their FP32 kinetic terms (u_y = u_z = 0: every operation rounds once): a
    large one, then n - 1 of about 2^-25 of it, below half a unit of its last place."""
    u = np.concatenate([[2.0], rng.uniform(1.1, 1.4, n - 1) * 2.0 ** -12]).astype(np.float32)
    one, u2 = np.float32(1), u * u
    return u, u2 / (np.sqrt(one + u2) + one)


@pytest.mark.parametrize("dims", [2, 3])
@pytest.mark.parametrize("n", [40, 300])
def test_kinetic_energy_sums_as_64_bits_do(dims, n):
    """n terms in one thread of the energy kernel, all others zero. (The kernel's threads take the records
    t, t + 256 blocks, ...; four blocks per SM at this many particles. n = 300 passes the point where the
    three FP32 numbers are added to an FP64 one.) An FP64 sum of n terms is within n 2^-53 of the exact one, and
    two roundings follow: the bound is (n + 8) 2^-53, 2^-44.7 at n = 300. FP32 terms summed into two FP32 numbers miss it
    (checked here), as the second one rounds at 2^-43 and above."""
    rng = np.random.default_rng(n)
    u, t = _terms(rng, n)
    exact = math.fsum(t.tolist())
    tol = (n + 8) * 2.0 ** -53
    s = c = np.float32(0)
    for x in t:
        y = np.float32(s + x)
        b = np.float32(y - s)
        c = np.float32(c + np.float32(np.float32(s - np.float32(y - b)) + np.float32(x - b)))
        s = y
    assert abs((float(s) + float(c)) / exact - 1) > tol        # the inputs can tell
    stride = 4 * 256 * torch.cuda.get_device_properties(0).multi_processor_count
    edge = 512 if dims == 2 else 64
    per_row = edge if dims == 2 else edge * edge
    ppc = -(-n * stride // (per_row * (edge // 2)))
    w = workload("transport", nx=edge, nz=edge, slab_k=edge // 2, ppc_ion=ppc, T_ion_K=0.0, **({} if dims == 2 else dict(
        dims=3, ny=edge)))
    sim = gb().Simulation(w)
    assert sim.info()["num_particles"][0] >= n * stride
    ck = sim.checkpoint()
    torch.cuda.synchronize()
    cap = sim.info()["num_particles"][0]
    slot = (4 * cap + 255) // 256 * 256                        # cell, fx, fz, u_x, ... behind a 256-byte header
    ux = ck[256 + 3 * slot:256 + 3 * slot + 4 * cap].view(torch.float32)
    assert not ux.any()
    e = []
    for m in (1, n):
        ux[5:5 + stride * m:stride] = torch.from_numpy(u[:m]).cuda()
        sim.restore(ck)
        e.append(sim.energy()["kinetic_ion"])
    assert abs(e[1] / e[0] / (exact / float(t[0])) - 1) <= tol
    sim.close()
