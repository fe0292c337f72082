"""The batched particle kernel's forms that the 16-cell tile with fields does not take: another tile (the window edge
at run time), tiles that differ between the slabs, the transport stage (no fields, currents or second set of
grids), with graphs of both parities and sorts in between. Grids bit for bit those of the slabs run alone."""
import pytest

from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_batch import gb, small_sweep  # noqa: F401
from tests.test_gpu_batch_state import _same_grids, _single

pytestmark = pytest.mark.gpu


def _atoms():
    return [workload("crater", nx=nx, nz=nz, slab_k=nz // 2, ppc_ion=ppc, seed=300 + nx)
            for nx, nz, ppc in ((48, 40, 16), (37, 51, 40), (131, 64, 9))]


@pytest.mark.parametrize("mode", ["full", "transport"])
@pytest.mark.parametrize("tiles", [(12, 12, 12), (12, 16, 20), (16, 16, 16)])
def test_batch_of_other_tiles_equals_single_runs(gb, mode, tiles):  # noqa: F811
    ws = [dict(w, tile=t) for w, t in zip(small_sweep() if mode == "full" else _atoms(), tiles)]
    batch = gb.Batch(ws, sort_every=4)
    batch.step(3)
    batch.step(6)
    for i, w in enumerate(ws):
        single = _single(gb, w, 9, sort_every=4)
        _same_grids(batch.slabs[i], single)
        single.close()
    batch.close()
