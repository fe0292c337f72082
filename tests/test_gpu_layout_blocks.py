"""The sort's storage layout where its block follows the particles per cell (2^17 particles and more):
32 x the particles per cell, the nearest power of two from 256 to 4096. The storage order is undone on the
host with that block and must be the cell order of every tile; a step from it deposits exactly what the
moved particles deposit afresh."""
import numpy as np
import pytest

from paper_1502_07722_gb300.workloads import workload
from tests.sort_layout import cell_key, undo_layout
from tests.test_gpu_layout import gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ppc,block", [(2, 3, 256), (2, 8, 256), (2, 13, 512), (2, 32, 1024), (2, 47, 2048),
                                            (2, 128, 4096), (2, 300, 4096), (3, 8, 256), (3, 16, 512)])
def test_layout_block_follows_the_load(gb, dims, ppc, block):  # noqa: F811
    ny = 11 if dims == 3 else 1
    nz = 40
    nx = -(-140000 // (20 * ppc * ny)) | 1
    w = dict(workload("transport"), nx=nx, nz=nz, slab_k=20, ppc_ion=ppc)
    if dims == 3:
        w.update(dims=3, ny=ny)
    T = 10 if dims == 3 else 16
    sim = gb.Simulation(w, sort_every=0)
    assert sim.info()["num_particles"][0] >= 1 << 17
    for _ in range(2):
        cell = sim.get_particles(0)["cell"].cpu().numpy().astype(np.int64)
        ordered, starts = undo_layout(cell_key(cell, nx, ny, T, dims), T ** dims, block)
        for a, b in zip(starts[:-1], starts[1:]):
            assert (np.diff(ordered[a:b]) >= 0).all()
        sim.step(3)
        rho, _ = sim.deposit_density()
        assert np.array_equal(sim.get_density().cpu().numpy(), rho.cpu().numpy())
        sim.sort()          # tiles of uneven counts, starting anywhere
    sim.close()
