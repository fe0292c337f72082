"""A batch whose slabs' state is written from outside between its steps goes on as the same slabs run alone do.
Every grid bit for bit: the deposits are exact integers whatever the particles' order."""
import pytest

from tests.test_gpu_batch import _state, gb, small_sweep  # noqa: F401

pytestmark = pytest.mark.gpu


def _same_grids(a, b):
    a, b = _state(a), _state(b)
    for x, y in zip((a[0], a[1], *a[2]), (b[0], b[1], *b[2])):
        assert (x == y).all()


def _single(gb, w, n, **over):
    sim = gb.Simulation(w, **over)
    sim.step(n)
    return sim


@pytest.mark.parametrize("sort_every", [0, 3])
def test_restored_slab_is_at_its_own_step(gb, sort_every):  # noqa: F811
    """One slab goes back to step 3, near the pulse's peak (steps 5 and on), while the others stay at 6:
    each goes on with the laser phase of its own step."""
    ws = small_sweep()
    batch = gb.Batch(ws, sort_every=sort_every)
    batch.step(3)
    ck = batch.slabs[1].checkpoint()
    batch.step(3)
    batch.slabs[1].restore(ck)
    batch.step(4)
    for i, n in enumerate((10, 7, 10)):
        assert batch.slabs[i].info()["step"] == n
        single = _single(gb, ws[i], n, sort_every=sort_every)
        _same_grids(batch.slabs[i], single)
        single.close()
    batch.close()


def test_slab_sorted_on_its_own(gb):  # noqa: F811
    """The sort leaves the slab's particles in its second buffers; the batch moves those, and its own sorts (every 5
    steps) go on from them."""
    ws = small_sweep()
    batch = gb.Batch(ws, sort_every=5)
    batch.step(4)
    batch.slabs[1].sort()
    batch.step(7)
    for i in range(3):
        fresh, _ = batch.slabs[i].deposit_density()
        assert fresh.equal(batch.slabs[i].get_density())
        single = _single(gb, ws[i], 11, sort_every=5)
        _same_grids(batch.slabs[i], single)
        single.close()
    batch.close()
