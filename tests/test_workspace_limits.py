"""The largest grids keep one set of field and current grids (64 bytes per node, 8 per cell for the sort, one more for
everything else): a state that filled the GPU with one set needs no second one. Smaller states have both."""
import ctypes

import paper_1502_07722_gb300 as gb
from paper_1502_07722_gb300 import _build
from paper_1502_07722_gb300.workloads import workload


def _sparse(nx, nz, **over):
    return gb.make_config(workload("tiny", nx=nx, nz=nz, slab_k=1, ppc_ion=1, ppc_electron=1, **over))


def test_largest_grids_have_one_set():
    _build.build()
    n2 = 32767 * 32768
    assert gb.pic_workspace_size(_sparse(32767, 32767)) < 73 * n2
    n3 = 1290 * 1290 * 1290
    assert n3 < 2 ** 31
    assert gb.pic_workspace_size(_sparse(1290, 1289, dims=3, ny=1290)) < 74 * n3
    half = _sparse(16320, 32766)
    assert gb.pic_workspace_size(half) > 112 * 16320 * 32767
    assert gb.pic_batch_workspace_size([half, half]) < 2 * 73 * 16320 * 32767


def test_list_of_work_items_is_small():
    """One entry (32 bytes) per tile and per 256 particles: with the smallest tiles 8 bytes per cell."""
    _build.build()
    n = ctypes.c_size_t()
    cfg = gb.make_config(workload("transport", nx=4096, nz=4096, slab_k=1, ppc_ion=1, tile=2))
    assert gb.load_library().pic_workspace_size(ctypes.byref(cfg), ctypes.byref(n)) == gb.PIC_OK
    assert n.value < (64 + 8 + 8 + 4) * 4096 * 4097
