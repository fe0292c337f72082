"""States too large for a second set of grids (kTwinBytes, 112 GiB with it): the field update in place. A slab of 64 columns
repeated over the whole width, particles, fields and plane-wave pulse alike, keeps the same bits in every repetition
as the slab alone, which has two sets. 2D, 3D and a batch of two; about 80 GB each."""
import pytest

from paper_1502_07722_gb300.workloads import workload

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gb():
    if not torch.cuda.is_available() or torch.cuda.mem_get_info()[1] < 200e9:
        pytest.skip("needs a GPU with 200 GB")
    from paper_1502_07722_gb300 import _build
    _build.build()
    import paper_1502_07722_gb300 as m
    yield m
    torch.cuda.empty_cache()


PERIOD = 64


def _config(nx, ny, nz):
    rows, ppc = (4, 2) if ny == 0 else (1, 1)
    w = workload("tiny", nx=nx, nz=nz, slab_k=rows, ppc_ion=ppc, ppc_electron=ppc, t_peak=0.0, tau_fwhm=1e-13)
    return w if ny == 0 else dict(w, dims=3, ny=ny)


def _fill(sim, w, seed):
    """The same particles and fields in every period (drawn on the device: 64 columns, and 64 rows in 3D, per period)."""
    g = torch.Generator("cuda")
    g.manual_seed(seed)
    d3 = "ny" in w
    py = PERIOD if d3 else 1
    rx, ry = w["nx"] // PERIOD, w["ny"] // py if d3 else 1
    rows = w["slab_k"]
    n = w["ppc_ion"] * PERIOD * py * rows
    for s in (0, 1):
        i, j, k = (torch.randint(0, m, (n,), generator=g, device="cuda") for m in (PERIOD, py, rows))
        f = [torch.rand(n, generator=g, device="cuda") * 0.999 for _ in range(3)]
        u = [torch.randn(n, generator=g, device="cuda") * (1e-4, 2e-2)[s] for _ in range(3)]
        a = torch.arange(rx, device="cuda").view(1, rx, 1) * PERIOD
        b = torch.arange(ry, device="cuda").view(ry, 1, 1) * py
        cell = ((k * py * ry + j + b) * w["nx"] + i + a).reshape(-1).int()
        many = lambda v: v.expand(ry, rx, n).reshape(-1).contiguous()  # noqa: E731
        sim.set_particles(s, cell, many(f[0]), many(f[2]), *map(many, u), fy=many(f[1]) if d3 else None)
    for q in range(6):
        one = torch.randn((w["nz"] + 1, py, PERIOD), generator=g, device="cuda") * (1e9 if q < 3 else 3.0)
        one = one.view(w["nz"] + 1, 1, py, 1, PERIOD).expand(-1, ry, -1, rx, -1).reshape(-1)
        sim.set_field(q, one)
        del one


def _compare(small, big, w):
    py = PERIOD if "ny" in w else 1
    shape = (w["nz"] + 1, -1, py, w["nx"] // PERIOD, PERIOD)
    one = (w["nz"] + 1, 1, py, 1, PERIOD)
    for get in [lambda s: s.get_density()] + [lambda s, q=q: s.get_field(q) for q in range(6)]:
        a, b = get(small).view(one), get(big).view(shape)
        assert bool((a == b).all())
        del a, b


@pytest.mark.parametrize("nx,ny,nz", [(32704, 0, 32767), (8192, 4096, 30)])
def test_in_place_update_equals_the_other(gb, nx, ny, nz):
    w, ws = _config(nx, ny, nz), _config(PERIOD, PERIOD if ny else 0, nz)
    nodes = nx * max(ny, 1) * (nz + 1)
    assert gb.pic_workspace_size(gb.make_config(w)) < 80 * nodes < 112 * nodes       # one set
    big, small = gb.Simulation(w, sort_every=2), gb.Simulation(ws, sort_every=2)
    for sim, c in ((big, w), (small, ws)):
        _fill(sim, c, 5)
        sim.step(3)
    _compare(small, big, w)
    big.close()
    small.close()


def test_batch_in_place(gb):
    ws = [_config(16320, 0, 32766), _config(16320, 0, 32700)]
    batch = gb.Batch(ws, sort_every=2)
    for sl, w in zip(batch.slabs, ws):
        _fill(sl, w, w["nz"])
    batch.step(3)
    for sl, w in zip(batch.slabs, ws):
        c = _config(PERIOD, 0, w["nz"])
        small = gb.Simulation(c, sort_every=2)
        _fill(small, c, w["nz"])
        small.step(3)
        _compare(small, sl, w)
        small.close()
    batch.close()
