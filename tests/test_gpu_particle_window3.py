"""One full step of the 3D particle kernel against the oracle where the staged window can go wrong: grids
narrower than the 13-node window (x, y wrap inside it), one column more and less, ragged tiles, and
electrons crossing cell edges both ways in every direction. Positions to 1e-5 of the displacement plus
the rounding of the offset; currents and density bit-exact against the oracle's deposits of the
GPU's own move (the tolerances of the one-step 3D parity)."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_3d import gb, random_state, set_both3, to_global3, w3  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,tile", [(4, 3, 5, 10), (12, 13, 9, 10), (13, 12, 11, 10), (31, 11, 21, 10), (9, 22, 8, 6)])
def test_one_step3_on_ragged_windows(gb, nx, ny, nz, tile):  # noqa: F811
    slab = max(2, nz // 2)
    w = w3(nx=nx, ny=ny, nz=nz, slab_k=slab, max_particles=20000, sort_every=0, tile=tile)
    sim = gb.Simulation(w)
    orc = oracle.Oracle3D(w, with_particles=False)
    g0 = []
    for sp, spread in ((0, 2e-4), (1, 3e-3)):
        x, y, z, u = random_state(40 + sp, nx, ny, nz, slab, 3000, spread)
        if sp:
            for d in range(3):
                u[d][d::9] = 0.3
                u[d][d + 3::9] = -0.3
        g0.append(set_both3(sim, orc, sp, x, y, z, u))
    sim.step(1)
    orc.step(1)
    J = np.zeros((3, nz + 1, ny, nx), np.int64)
    for sp, sign in ((0, 1), (1, -1)):
        X1, Y1, Z1, U1 = to_global3(sim.get_particles(sp), nx, ny)
        X0, Y0, Z0, _ = to_global3(g0[sp], nx, ny)
        o = orc.get_particles(sp)
        for a, b, a0, n in ((X1, o["x"], X0, nx), (Y1, o["y"], Y0, ny)):
            d = np.abs(np.mod(a - b + n / 2, n) - n / 2)
            disp = np.abs(np.mod(b - a0 + n / 2, n) - n / 2)
            assert (d <= 1e-5 * disp + 2.0 ** -22).all()
        assert (np.abs(Z1 - o["z"]) <= 1e-5 * np.abs(o["z"] - Z0) + 2.0 ** -22).all()
        for c, key in enumerate(("ux", "uy", "uz")):
            np.testing.assert_allclose(U1[c], o[key], rtol=1e-5, atol=1e-6 * np.abs(o[key]).max())
        oracle.deposit_current3(nx, ny, nz, sign, X0, Y0, Z0, X1, Y1, Z1, out=J)
    assert np.array_equal(sim.get_current().cpu().numpy(), J)
    X1, Y1, Z1, _ = to_global3(sim.get_particles(0), nx, ny)
    assert np.array_equal(sim.get_density().cpu().numpy(), oracle.deposit_density3(nx, ny, nz, X1, Y1, Z1))
    sim.close()
