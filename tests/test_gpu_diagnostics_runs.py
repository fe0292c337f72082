"""The diagnostics that sum runs of particles of one cell in registers (density deposit, cell moments) and the
two-sum energies, in the states where that can go wrong: storage order far from the cell order (many steps
without a sort), one particle, fewer than a warp, a particle count around a multiple of a warp's chunk,
momenta whose squares leave FP32's range. Density: bit for bit the oracle's deposit. Temperature: FP64
sums per cell on the host, 1e-12 of the cell's mean square momentum (three FP32 numbers carry more than
2^-60, the host sums about 1e-15). Kinetic energy: the FP64 energy within the rounding of the FP32 terms, 4 x 2^-24."""
import numpy as np
import pytest

import oracle
from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_parity import _built, gb, to_global  # noqa: F401

pytestmark = pytest.mark.gpu
C, KB, AMU = 299792458.0, 1.380649e-23, 1.66053906660e-27


@pytest.mark.parametrize("n,scale,order", [(1, 1e-3, "any"), (31, 1e-3, "any"), (1000, 1e-6, "any"), (1025, 1e-3, "drift"),
                                           (40000, 1e-3, "drift"), (200001, 1e-3, "drift"), (3000, 1e17, "any")])
def test_runs_and_sums(n, scale, order):
    nx, nz = 37, 26
    w = workload("transport", nx=nx, nz=nz, slab_k=13, ppc_ion=1, max_particles=max(n, 13 * nx),
                 dt_override=6e-16, D_eV=1e-18)          # positions drift freely
    sim = gb().Simulation(w, sort_every=0)
    rng = np.random.default_rng(n)
    cell = rng.integers(0, nx * nz, n).astype(np.int32)
    f = [rng.random(n, dtype=np.float32) * np.float32(0.999) for _ in range(2)]
    u = [rng.normal(0, scale, n).astype(np.float32) for _ in range(3)]
    sim.set_particles(0, cell, f[0], f[1], *u)
    if order == "drift":
        sim.step(90)                           # the storage order now mixes cells
    p = sim.get_particles(0)
    x, z, v = to_global(p, nx)
    rho, _ = sim.deposit_density()
    assert np.array_equal(rho.cpu().numpy(), oracle.deposit_density(nx, nz, x, z))
    c = p["cell"].cpu().numpy()
    num = np.bincount(c, minlength=nx * nz).astype(np.float64)
    s1 = [np.bincount(c, q, nx * nz) for q in v]
    s2 = np.bincount(c, v[0] ** 2 + v[1] ** 2 + v[2] ** 2, nx * nz)
    m = w["ion_mass_amu"] * AMU * C * C / (3 * KB)
    ok = num >= 2
    T = np.zeros(nx * nz)
    T[ok] = m * (s2 - sum(q ** 2 for q in s1) / np.maximum(num, 1))[ok] / (num[ok] - 1)
    got = sim.cell_temperature(0).cpu().numpy().reshape(-1)
    tol = 1e-12 * m * s2 / np.maximum(num - 1, 1)
    assert (np.abs(got - T) <= tol).all()
    if scale < 1:
        a = [p[q].cpu().numpy() for q in ("ux", "uy", "uz")]
        u2 = sum(q.astype(np.float64) ** 2 for q in a)
        ke = (u2 / (np.sqrt(1 + u2) + 1)).sum() * sim.info()["weight"] * w["ion_mass_amu"] * AMU * C * C
        assert abs(sim.energy()["kinetic_ion"] / ke - 1) < 4 * 2.0 ** -24      # the FP32 terms' own rounding
    sim.close()
