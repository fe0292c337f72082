"""Periodic grids narrower than the particle kernels' window: one tile or two, whose window holds some columns
twice. The same slab repeated side by side on a wide grid, where every column is in the window once, has the same
fields, currents and density in every repetition, bit for bit (a particle outside the window would gather its fields another
way)."""
import numpy as np
import pytest

from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_parity import _built, gb  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _particles(rng, nx, ny, nz, rows, n, spread):
    i, j, k = rng.integers(0, nx, n), rng.integers(0, ny, n), rng.integers(0, rows, n)
    f = [rng.random(n, dtype=np.float32) * np.float32(0.999) for _ in range(3)]
    u = [rng.normal(0, spread, n).astype(np.float32) for _ in range(3)]
    return (i, j, k), f, u


def _run(w, ny, reps, sets, fields, steps):
    """reps copies along x (and along y in 3D) of the particle sets and fields of one period."""
    nx, nz, d3 = w["nx"], w["nz"], "ny" in w
    ry = reps if d3 else 1
    big = dict(w, nx=nx * reps, max_particles=max(s[0][0].size for s in sets) * reps * ry)
    if d3:
        big["ny"] = ny * reps
    sim = gb().Simulation(big, sort_every=0)
    for s, ((i, j, k), f, u) in enumerate(sets):
        cells = [((k * ny * ry + j + b * ny) * nx * reps + i + a * nx) for b in range(ry) for a in range(reps)]
        many = lambda v: np.concatenate([v] * (reps * ry))  # noqa: E731
        sim.set_particles(s, np.concatenate(cells).astype(np.int32), many(f[0]), many(f[2]), *map(many, u),
                          fy=many(f[1]) if d3 else None)
    for q, v in enumerate(fields):
        sim.set_field(q, np.tile(v, (1, ry, reps)) if d3 else np.tile(v[:, 0], (1, reps)))
    sim.step(steps)
    shape = (nz + 1, ry, ny, reps, nx)
    out = [sim.get_density(), *sim.get_current(), *(sim.get_field(q) for q in range(6))][:None if sim.nspecies > 1 else 1]
    out = [o.reshape(shape) for o in out]
    sim.close()
    return out


@pytest.mark.parametrize("mode", ["full", "transport"])
@pytest.mark.parametrize("dims,nx,ny", [(2, 3, 1), (2, 12, 1), (2, 16, 1), (2, 17, 1), (2, 18, 1), (2, 19, 1), (3, 10, 10),
                                        (3, 8, 24), (3, 24, 9), (3, 11, 12), (3, 3, 4)])
def test_narrow_grid_equals_its_repetitions(mode, dims, nx, ny):
    rng = np.random.default_rng(nx * 100 + ny)
    nz, rows = 24, 12
    n = 4 * nx * ny * rows
    w = workload("tiny" if mode == "full" else "transport", nx=nx, nz=nz, slab_k=rows, ppc_ion=4,
                 ppc_electron=4 if mode == "full" else 0, **(dict(dims=3, ny=ny) if dims == 3 else {}))
    sets = [_particles(rng, nx, ny, nz, rows, n, 1e-4)]
    fields = [np.zeros((nz + 1, ny, nx), np.float32)] * 6
    if mode == "full":
        sets.append(_particles(rng, nx, ny, nz, rows, n, 5e-2))
        fields = [rng.normal(0, 1e9 if q < 3 else 3.0, (nz + 1, ny, nx)).astype(np.float32) for q in range(6)]
    reps = 8 if nx < 8 or ny < 8 and dims == 3 else 4
    one, many = _run(w, ny, 1, sets, fields, 3), _run(w, ny, reps, sets, fields, 3)
    for a, b in zip(one, many):
        assert torch.equal(a.expand_as(b), b)
