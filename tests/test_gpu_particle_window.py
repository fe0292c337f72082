"""One full step of the 2D particle kernel against the oracle where the staged window can go wrong:
grids narrower than the window (x wraps inside it), one column more and less than it, ragged tiles, the
compiled-in window edge (16-cell tiles) and the run-time one. Particles near the seam, the walls, on nodes
and crossing cell edges; currents and density bit-exact against the oracle's deposits of the GPU's own
move. Tolerance: that of the one-step particle parity."""
import numpy as np
import pytest

import oracle
from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_parity import _built, _compare_particles, _random_state, gb, set_both, to_global  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,tile", [(4, 5, 16), (17, 9, 16), (22, 40, 16), (23, 18, 16), (24, 17, 16), (49, 33, 16),
                                        (45, 33, 8), (11, 30, 8), (61, 48, 20)])
def test_one_step_on_ragged_windows(nx, nz, tile):
    sk = max(2, nz // 2)
    w = workload("tiny", nx=nx, nz=nz, slab_k=sk, max_particles=8 * nx * sk, I0=1e19, tile=tile)
    sim = gb().Simulation(w, sort_every=0)
    orc = oracle.Oracle(w, with_particles=False)
    ions, els, fields = _random_state(nx, nz, sk, 9, w)
    # electrons that cross a cell edge in the step, left and right
    els["ux"][::7] = 0.3
    els["ux"][3::7] = -0.3
    els["uz"][1::5] = 0.25
    g0 = [set_both(sim, orc, 0, ions), set_both(sim, orc, 1, els)]
    for f, a in enumerate(fields):
        sim.set_field(f, a)
        orc.set_field(f, a)
    sim.step(1)
    orc.step(1)
    g1 = [sim.get_particles(s) for s in (0, 1)]
    for sp in (0, 1):
        _compare_particles(g1[sp], orc.get_particles(sp), g0[sp], nx)
    J = np.zeros((3, nz + 1, nx), np.int64)
    for sp, sign in ((0, 1), (1, -1)):
        x0, z0, _ = to_global(g0[sp], nx)
        x1, z1, u1 = to_global(g1[sp], nx)
        oracle.deposit_current(nx, nz, sign, x0, z0, x1, z1, *[v.astype(np.float32) for v in u1], out=J, bits=18)
    assert np.array_equal(sim.get_current().cpu().numpy(), J)
    x1, z1, _ = to_global(g1[0], nx)
    assert np.array_equal(sim.get_density().cpu().numpy(), oracle.deposit_density(nx, nz, x1, z1))
    sim.close()
