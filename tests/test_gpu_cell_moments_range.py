"""Cell temperatures of momenta whose squares leave FP32's range downwards, alone and beside ordinary ones. The FP32
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
