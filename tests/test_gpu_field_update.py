"""The one-kernel Yee update at the sizes where its work split can go wrong: grids narrower than a
warp's 29 columns, one column more or less than a multiple of them, row counts around multiples of
the 4-row segments. Fields against the oracle's Maxwell step from the same fields and the GPU's own
current; the density and the current of a later step bit-exact against the oracle's deposits of the
GPU's own moves, which holds only when the step before cleared the currents and started the
density. Tolerances: those of the one-step field parity (1e-5 relative, 1e-6 of the field's maximum)."""
import numpy as np
import pytest

import oracle
from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_parity import _built, _random_state, gb, set_both, to_global  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("laser", [1, 0])
@pytest.mark.parametrize("nx,nz", [(3, 4), (5, 5), (28, 7), (29, 8), (30, 9), (58, 10), (59, 11), (87, 12), (88, 35)])
def test_field_update_on_ragged_grids(nx, nz, laser):
    sk = max(1, nz // 2)
    w = workload("tiny", nx=nx, nz=nz, slab_k=sk, max_particles=8 * nx * sk, I0=1e19, laser_profile=laser)
    sim = gb().Simulation(w, sort_every=0)
    orc = oracle.Oracle(w, with_particles=False)
    ions, els, fields = _random_state(nx, nz, sk, 3, w)
    set_both(sim, orc, 0, ions)
    set_both(sim, orc, 1, els)
    for f, a in enumerate(fields):
        sim.set_field(f, a)
    for step in range(1 if laser else 3):
        g0 = [sim.get_particles(s) for s in (0, 1)]
        F0 = [sim.get_field(f).cpu().numpy().astype(np.float64) for f in range(6)]
        sim.step(1)
        g1 = [sim.get_particles(s) for s in (0, 1)]
        J = np.zeros((3, nz + 1, nx), np.int64)
        for sp, sign in ((0, 1), (1, -1)):
            x0, z0, _ = to_global(g0[sp], nx)
            x1, z1, u1 = to_global(g1[sp], nx)
            oracle.deposit_current(nx, nz, sign, x0, z0, x1, z1, *[v.astype(np.float32) for v in u1], out=J, bits=18)
        assert np.array_equal(sim.get_current().cpu().numpy(), J)
        x1, z1, _ = to_global(g1[0], nx)
        assert np.array_equal(sim.get_density().cpu().numpy(), oracle.deposit_density(nx, nz, x1, z1))
        fo = oracle.Oracle(w, with_particles=False)
        for f, a in enumerate(F0):
            fo.set_field(f, a)
        fo.set_current(J)
        fo.maxwell()
        for f in range(6):
            b = fo.get_field(f)
            np.testing.assert_allclose(sim.get_field(f).cpu().numpy(), b, rtol=1e-5, atol=1e-6 * np.abs(b).max())
    sim.close()


def test_state_written_between_steps_prepares_the_next_one():
    """A checkpoint restored after some steps, and new particles, invalidate what the field update
    prepared: the run after them equals a fresh context's bit for bit."""
    w = workload("tiny", nx=45, nz=26, slab_k=13)
    a, b = gb().Simulation(w, sort_every=0), gb().Simulation(w, sort_every=0)
    ck = a.checkpoint()
    a.step(3)
    a.restore(ck)
    a.step(2)
    b.restore(ck)
    b.step(2)
    for s in (0, 1):
        p = b.get_particles(s)
        for sim in (a, b):
            sim.set_particles(s, **p)
    a.step(2)
    b.step(2)
    assert np.array_equal(a.get_density().cpu().numpy(), b.get_density().cpu().numpy())
    assert np.array_equal(a.get_current().cpu().numpy(), b.get_current().cpu().numpy())
    for f in range(6):
        assert np.array_equal(a.get_field(f).cpu().numpy(), b.get_field(f).cpu().numpy())
    a.close()
    b.close()
