"""Cell temperatures of momenta whose squares leave FP32's range, alone and beside ordinary ones. The FP32
products of the kernel's three-number sums are exact down to 2^-40 per momentum; smaller ones are summed in FP64. Against
FP64 sums on the host, 1e-12 of the cell's mean square momentum, as for ordinary momenta."""
import numpy as np
import pytest

from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_diagnostics_runs import AMU, C, KB
from tests.test_gpu_parity import _built, gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-12, 1e-14, 1e-17, 1e-20, 1e-25, 1e-30])
@pytest.mark.parametrize("mixed", [False, True])
def test_small_momenta(scale, mixed):
    nx, nz, n = 19, 12, 4000
    w = workload("transport", nx=nx, nz=nz, slab_k=6, ppc_ion=1, max_particles=n)
    sim = gb().Simulation(w, sort_every=0)
    rng = np.random.default_rng(3)
    cell = rng.integers(0, nx * nz, n).astype(np.int32)
    f = rng.random(n, dtype=np.float32) * np.float32(0.999)
    size = np.where(rng.random(n) < 0.5, scale, 1e-4) if mixed else scale
    u = [(rng.normal(0, 1, n) * size).astype(np.float32) for _ in range(3)]
    u[0][::7] = u[1][::7] = u[2][::7] = 0
    sim.set_particles(0, cell, f, f, *u)
    p = sim.get_particles(0)
    c = p["cell"].cpu().numpy()
    v = [p[k].cpu().numpy().astype(np.float64) for k in ("ux", "uy", "uz")]
    num = np.bincount(c, minlength=nx * nz).astype(np.float64)
    s2 = np.bincount(c, v[0] ** 2 + v[1] ** 2 + v[2] ** 2, nx * nz)
    ok = num >= 2
    m = w["ion_mass_amu"] * AMU * C * C / (3 * KB)
    T = np.where(ok, m * (s2 - sum(np.bincount(c, q, nx * nz) ** 2 for q in v) / np.maximum(num, 1)) /
                 np.maximum(num - 1, 1), 0.0)
    got = sim.cell_temperature(0).cpu().numpy().reshape(-1)
    assert (np.abs(got - T) <= 1e-12 * m * s2 / np.maximum(num - 1, 1)).all()
    sim.close()


@pytest.mark.parametrize("order", ["sorted", "shuffled"])
@pytest.mark.parametrize("dims,ppc", [(2, 47), (2, 8), (3, 64), (2, 9), (2, 1)])
def test_large_states_of_any_order_and_size_of_momenta(dims, ppc, order):
    """Above the particle count from which runs of one cell are walked (with 47, 8 and 64 per cell; 9 and 1 take one
    reduction per particle): momenta from 1e-30 to 1e17, a size per cell and every fifth particle of another,
    stored in the order of the sort and at random."""
    import torch
    nx, ny, nz = (257, 1, 2 * -(-(5 << 18) // (257 * ppc))) if dims == 2 else (41, 37, 2 * -(-(7 << 18) // (41 * 37 * ppc)))
    w = workload("transport", nx=nx, nz=nz, slab_k=nz // 2, ppc_ion=ppc, T_ion_K=0.0, **({} if dims == 2 else dict(dims=3, ny=ny)))
    sim = gb().Simulation(w, sort_every=0)
    n, ncell = sim.info()["num_particles"][0], nx * ny * nz
    assert n > (1 << 20 if dims == 2 else 3 << 19)
    ck = sim.checkpoint()
    torch.cuda.synchronize()
    slot = (4 * n + 255) // 256 * 256
    part = lambda q, t: ck[256 + q * slot:256 + q * slot + 4 * n].view(t)  # noqa: E731
    rng = np.random.default_rng(ppc)
    c = part(0, torch.int32).cpu().numpy()
    if order == "shuffled":
        c = rng.permutation(c)
        part(0, torch.int32).copy_(torch.from_numpy(c))
    size = 10.0 ** rng.integers(-30, 18, ncell)
    size = np.where(np.arange(n) % 5 == 0, 1e-6 * size[c], size[c])
    v = []
    for q in (3, 4, 5):
        u = (rng.normal(0, 1, n) * size).astype(np.float32)
        part(q, torch.float32).copy_(torch.from_numpy(u))
        v.append(u.astype(np.float64))
    sim.restore(ck)
    num = np.bincount(c, minlength=ncell).astype(np.float64)
    s2 = np.bincount(c, v[0] ** 2 + v[1] ** 2 + v[2] ** 2, ncell)
    m = w["ion_mass_amu"] * AMU * C * C / (3 * KB)
    T = np.where(num >= 2, m * (s2 - sum(np.bincount(c, q, ncell) ** 2 for q in v) / np.maximum(num, 1)) /
                 np.maximum(num - 1, 1), 0.0)
    got = sim.cell_temperature(0).cpu().numpy().reshape(-1)
    assert (np.abs(got - T) <= 1e-12 * m * s2 / np.maximum(num - 1, 1)).all()
    sim.close()
