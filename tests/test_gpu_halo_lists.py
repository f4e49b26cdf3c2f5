"""Where the halo schedule's lists go when the interface arrays leave no room:
contexts created with the exact number of interface cells, and dense media."""
import numpy as np
import pytest

from paper_2009_12584_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2009_12584_gb300 import lbm  # noqa: E402

IMPROVED = ("virtual_avg", dict(G_s=(3.0, 3.0), chi=(1.2, 0.8)))
LLKC = ("llkc", dict(G_s=(-0.5, 0.3)))


def _interface_cells(mask, per_x, per_y):
    """Solid nodes with a fluid D2Q9 neighbour (walls on the other borders)."""
    p = np.pad(mask, 1, constant_values=1)
    if per_x:
        p[:, 0], p[:, -1] = p[:, -2], p[:, 1]
    if per_y:
        p[0], p[-1] = p[-2], p[1]
    ny, nx = mask.shape
    near = np.zeros((ny, nx), bool)
    for dy in (0, 1, 2):
        for dx in (0, 1, 2):
            near |= p[dy:dy + ny, dx:dx + nx] == 0
    return int(((mask != 0) & near).sum())


def _masks():
    open_box = inputs.flat_wall_mask(200, 96)
    wells = np.ones((66, 99), np.uint8)
    wells[1::3, 1::3] = 0  # eight nodes in nine are interface cells (here the planes' padding holds their lists)
    return {"wall": open_box, "30%": inputs.random_solid_mask(131, 83, 1, 0.3),
            "45%": inputs.random_solid_mask(131, 83, 2, 0.45), "60%": inputs.random_solid_mask(131, 83, 3, 0.6),
            "wells": wells}


def _sim(mask, storage, kernel, wet, exact, seed=7):
    ny, nx = mask.shape
    per_y = bool((mask[0] == 0).any())
    cap = _interface_cells(mask, True, per_y) if exact else 0
    sim = lbm.Simulation(nx, ny, storage=storage, kernel=kernel, periodic_x=True, periodic_y=per_y, max_interface=cap)
    sim.set_geometry(mask).set_wetting(wet[0], **wet[1])
    if exact:
        assert sim.interface_count() == cap
    return sim.init_fields(*inputs.random_fields(nx, ny, seed, umax=0.05))


@pytest.mark.parametrize("storage,kernel", [("fp32", "auto"), ("fp32", "halo"), ("fp64", "halo")])
@pytest.mark.parametrize("wet", [IMPROVED, LLKC], ids=["improved", "llkc"])
@pytest.mark.parametrize("exact", [True, False])
@pytest.mark.parametrize("geometry", sorted(_masks()))
def test_lists_find_room(storage, kernel, wet, exact, geometry):
    """One launch per step, the bits of the two passes, and forces, moments and
    a restored state that leave the lists alone."""
    mask = _masks()[geometry]
    a = _sim(mask, storage, kernel, wet, exact)
    b = _sim(mask, storage, "two_pass", wet, exact)
    n0 = a.launch_count
    a.step(3)
    assert a.launch_count - n0 == 3
    b.step(3)
    assert torch.equal(a.forces(), b.forces())
    for x, y in zip(a.moments(), b.moments()):
        assert torch.equal(x, y)
    f = b.step(2).populations()
    assert torch.equal(a.step(2).populations(), f)
    a.set_populations(f)
    b.set_populations(f)
    a.set_wetting(*LLKC[:1], **LLKC[1])
    b.set_wetting(*LLKC[:1], **LLKC[1])
    assert torch.equal(a.step(2).populations(), b.step(2).populations())
    assert torch.equal(a.forces(), b.forces())
    a.sync()


@pytest.mark.parametrize("storage,kernel", [("fp32", "auto"), ("fp32", "halo"), ("fp64", "halo"), ("fp64", "auto")])
@pytest.mark.parametrize("graph", [0, 2])
def test_lists_give_way_to_batches(storage, kernel, graph):
    """Batch steps by either schedule, of odd and even number, between single
    steps, restored states and forces of members whose lists lie in a density
    plane."""
    masks = [_masks()[k] for k in ("wall", "45%", "30%")]
    wets = [IMPROVED, LLKC, IMPROVED]
    pairs = [(_sim(m, storage, kernel, w, True), _sim(m, storage, "two_pass", w, True)) for m, w in zip(masks, wets)]
    batch = lbm.Batch([p[0] for p in pairs])
    batch.set_graph_steps(graph)

    def check():
        for a, b in pairs:
            a.sync()
            assert torch.equal(a.populations(), b.populations())
            assert torch.equal(a.forces(), b.forces())
            for x, y in zip(a.moments(), b.moments()):
                assert torch.equal(x, y)

    def both(n, batched):
        batch.step(n) if batched else [a.step(n) for a, _ in pairs]
        for _, b in pairs:
            b.step(n)
        check()

    both(2, False)
    for schedule in ("two_pass", "tiled", "two_pass"):
        if schedule == "tiled" and kernel == "halo":
            continue  # no tile lists
        batch.set_schedule(schedule)
        both(3, True)
        both(2, False)
        both(4, True)
        for a, b in pairs:
            f = b.populations()
            a.set_populations(f)
            b.set_populations(f)
        both(1, True)
        # the halo launches are put together anew while the lists may be away
        for (a, b), (kind, kw) in zip(pairs, (LLKC, IMPROVED, LLKC)):
            a.set_wetting(kind, **kw)
            b.set_wetting(kind, **kw)
        both(2, True)
        if schedule == "tiled":
            batch.set_schedule("two_pass")
            both(3, True)
        both(1, False)
    batch.close()


@pytest.mark.parametrize("kernel,launches", [("auto", 2), ("halo", 3)])
def test_without_any_room(kernel, launches):
    """Eight nodes in nine are interface cells, on a grid with little padding:
    the lists fit nowhere. AUTO runs tiles (Eq. 8 and the tiles, after a first
    step that builds their lists and sums the densities), HALO the two passes."""
    nx, ny = 2016, 699
    mask = np.ones((ny, nx), np.uint8)
    mask[1::3, 1::3] = 0
    cap = _interface_cells(mask, True, True)
    sims = []
    for k, c in ((kernel, cap), ("two_pass", 0)):
        sim = lbm.Simulation(nx, ny, storage="fp32", kernel=k, periodic_x=True, periodic_y=True, max_interface=c)
        sim.set_geometry(mask).set_wetting(IMPROVED[0], **IMPROVED[1])
        sims.append(sim.init_fields(*inputs.random_fields(nx, ny, 3, umax=0.05)))
    a, b = sims
    a.step(1)
    n0 = a.launch_count
    a.step(2)
    assert a.launch_count - n0 == 2 * launches
    assert torch.equal(a.populations(), b.step(3).populations())
    assert torch.equal(a.moments()[0], b.moments()[0])
    assert torch.equal(a.step(2).populations(), b.step(2).populations())
