"""The reverse step from a checkpoint refuses a buffer that is none, or one of other species or particle counts, and leaves
the adjoints as they are. (No such call reaches a kernel: the header is checked on the host.)"""
import pytest

from paper_1502_07722_gb300 import diff
from paper_1502_07722_gb300.workloads import workload
from tests.test_gpu_adjoint import gb, small_full  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_reverse_step_from_a_foreign_buffer(gb):  # noqa: F811
    w = small_full()
    run = diff.DiffRun(w, w["D_eV"] * diff.QE, w["n_atoms"] ** (-1 / 3), w["I0"], every=4)
    weights = diff.crater_weights(w["nx"], w["nz"], w["slab_k"], w["dx"])
    run.forward(4, weights, 1e-3)
    bufs, grads = run._buffers(weights.numel())
    gb.pic_adjoint_seed(run.sim.h, 1e-3, weights.data_ptr(), bufs)
    bits = lambda t: t.view(torch.uint8)  # noqa: E731  (parts of the buffers are scratch)
    before = [t.clone() for t in run._keep]
    good = run.checkpoints[0]
    bad = [torch.zeros_like(good)]
    for at, value in ((0, 1), (16, 0), (24, 1 << 40), (32, 1 << 32 | 0)):      # magic, ion and electron counts, species
        b = good.clone()
        b[at:at + 8].view(torch.int64).fill_(value)
        bad.append(b)
    torch.cuda.synchronize()
    for b in bad:
        for call in (lambda: gb.pic_adjoint_step_at(run.sim.h, b.data_ptr(), bufs),
                     lambda: gb.pic_adjoint_steps_at(run.sim.h, [good.data_ptr(), b.data_ptr()], bufs)):
            with pytest.raises(gb.PicError) as e:
                call()
            assert e.value.code == gb.PIC_EINVAL
    torch.cuda.synchronize()
    for a, b in zip(before, run._keep):
        assert torch.equal(bits(a), bits(b))
    gb.pic_adjoint_step_at(run.sim.h, good.data_ptr(), bufs)          # the checkpoint itself is taken
    torch.cuda.synchronize()
    assert not torch.equal(bits(before[-1]), bits(run._keep[-1]))
    run.close()
