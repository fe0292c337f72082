"""The one-kernel 3D Yee update where its work split can go wrong: grids around multiples of its 29-column,
13-row patches and 16-plane segments, and smaller than one patch. Fields against the oracle's Maxwell step from
the same fields and the GPU's own current; currents and density of a later step bit-exact against the
oracle's deposits of the GPU's own moves (they hold only when the step before cleared the currents and
started the density). Tolerances: those of the one-step 3D parity."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_3d import gb, random_state, set_both3, to_global3, w3  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("laser", [1, 0])
@pytest.mark.parametrize("nx,ny,nz", [(3, 3, 4), (28, 12, 14), (29, 13, 15), (30, 14, 16), (58, 26, 30), (59, 27, 31),
                                      (31, 11, 32), (12, 40, 47)])
def test_field_update3_on_ragged_grids(gb, nx, ny, nz, laser):  # noqa: F811
    slab = max(1, nz // 2)
    w = w3(nx=nx, ny=ny, nz=nz, slab_k=slab, ppc_ion=1, ppc_electron=1, max_particles=100000, sort_every=0, tile=10,
           laser_profile=laser)
    sim = gb.Simulation(w)
    orc = oracle.Oracle3D(w, with_particles=False)
    for sp, spread in ((0, 2e-4), (1, 3e-3)):
        x, y, z, u = random_state(60 + sp, nx, ny, nz, slab, 2000, spread)
        set_both3(sim, orc, sp, x, y, z, u)
    rng = np.random.default_rng(8)
    for f in range(6):
        sim.set_field(f, rng.normal(0, 3e9 if f < 3 else 10.0, (nz + 1, ny, nx)).astype(np.float32))
    for step in range(1 if laser else 2):
        F0 = [sim.get_field(f).cpu().numpy().astype(np.float64) for f in range(6)]
        before = [to_global3(sim.get_particles(s), nx, ny) for s in (0, 1)]
        sim.step(1)
        after = [to_global3(sim.get_particles(s), nx, ny) for s in (0, 1)]
        J = np.zeros((3, nz + 1, ny, nx), np.int64)
        for s, sign in ((0, 1), (1, -1)):
            oracle.deposit_current3(nx, ny, nz, sign, *before[s][:3], *after[s][:3], out=J)
        assert np.array_equal(sim.get_current().cpu().numpy(), J)
        assert np.array_equal(sim.get_density().cpu().numpy(), oracle.deposit_density3(nx, ny, nz, *after[0][:3]))
        fo = oracle.Oracle3D(w, with_particles=False)
        for f in range(6):
            fo.set_field(f, F0[f])
        fo.set_current(J)
        fo.maxwell()
        for f in range(6):
            b = fo.get_field(f)
            np.testing.assert_allclose(sim.get_field(f).cpu().numpy(), b, rtol=1e-5, atol=1e-6 * np.abs(b).max())
    sim.close()
