"""A single run and the same slab in a batch drive the same field bit for bit, at steps where that hangs on the last
bit of the FP64 sine: its product with the amplitude lies next to a rounding boundary of FP32, and a host's sine
(glibc) falls on the other side of it than the device's. Found by a search over the first 2^34 steps of this run, whose
pulse is long enough to be flat over all of them."""
import pytest

from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_batch import gb  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("step", [5557176888, 7037528488, 9257930213, 9566246331])
def test_single_run_and_batch_take_the_same_antenna_field(gb, step):  # noqa: F811
    w = workload("tiny", tau_fwhm=1e-3)
    batch, sim = gb.Batch([w]), gb.Simulation(w)
    for s in (batch.slabs[0], sim):
        ck = s.checkpoint()
        torch.cuda.synchronize()
        ck[8:16].view(torch.int64).fill_(step)                # magic, step, ...
        torch.cuda.synchronize()
        s.restore(ck)
        assert s.info()["step"] == step
    batch.step(2)
    sim.step(2)
    a, b = batch.slabs[0].get_field(0), sim.get_field(0)
    assert a[62].abs().max() > 1e9 and torch.equal(a, b)
    batch.close()
    sim.close()
