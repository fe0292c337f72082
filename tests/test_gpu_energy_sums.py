"""What the energy sums take from a state: the electrons' momenta alone for their kinetic energy."""
import pytest

from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_parity import _built, gb  # noqa: F401
from tests.test_zz_no_alloc import _view

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_electron_cells_are_not_part_of_the_kinetic_energy():
    """A state view whose electron cells were never filled in (here -1): the same five energies."""
    sim = gb().Simulation(workload("tiny", nx=48, nz=40, slab_k=20))
    sim.step(3)
    view, keep = _view(gb(), sim)
    out = torch.empty((2, 5), dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream()
    gb().pic_energy_noalloc(sim.cfg, view, out[0].data_ptr(), st.cuda_stream)
    keep[1]["cell"].fill_(-1)
    gb().pic_energy_noalloc(sim.cfg, view, out[1].data_ptr(), st.cuda_stream)
    assert out[0, 1] > 0 and torch.equal(out[0], out[1])
    sim.close()
