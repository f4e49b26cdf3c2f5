"""Members of a batch that take another wetting scheme or geometry between
batch steps: from the next step on they step as alone."""
import pytest

from paper_2009_12584_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2009_12584_gb300 import lbm  # noqa: E402

SCHEMES = [("virtual_avg", dict(G_s=(3.0, 3.0), chi=(1.2, 0.8))), ("martys_chen", dict(G_s=(-0.2, 0.2))),
           ("virtual_avg", dict(G_s=(2.5, 3.5), chi=(0.9, 1.3), avg_stencil=9)), ("llkc", dict(G_s=(-0.5, 0.3)))]
SIZES = [(200, 90), (130, 101), (96, 64)]


@pytest.mark.parametrize("storage,kernel", [("fp32", "auto"), ("fp16", "auto"), ("fp32", "two_pass"), ("fp64", "auto")])
@pytest.mark.parametrize("schedule,graph", [("two_pass", 0), ("two_pass", 2), ("tiled", 2)])
def test_members_may_change_scheme_and_geometry(storage, kernel, schedule, graph):
    """Improved scheme to one-ring schemes and back (halo launches of one ring
    and of three, Eq. 8 blocks), then a geometry with more and one with fewer
    fluid nodes."""
    if schedule == "tiled" and (storage == "fp16" or kernel == "two_pass"):
        pytest.skip("no tiled batches")
    pairs = []
    for i, (nx, ny) in enumerate(SIZES):
        two = []
        for _ in range(2):
            sim = lbm.Simulation(nx, ny, storage=storage, kernel=kernel, periodic_x=True, periodic_y=True)
            sim.set_geometry(inputs.random_solid_mask(nx, ny, seed=i, fraction=0.04))
            sim.set_wetting(SCHEMES[i][0], **SCHEMES[i][1])
            two.append(sim.init_fields(*inputs.random_fields(nx, ny, 3 + i, umax=0.05)))
        pairs.append(two)
    batch = lbm.Batch([p[0] for p in pairs])
    batch.set_schedule(schedule)
    batch.set_graph_steps(graph)

    def check(n):
        batch.step(n)
        for a, b in pairs:
            b.step(n)
            a.sync()
            assert torch.equal(a.populations(), b.populations())

    check(3)
    for shift in (1, 2, 3):
        for i, p in enumerate(pairs):
            kind, kw = SCHEMES[(i + shift) % len(SCHEMES)]
            for sim in p:
                sim.set_wetting(kind, **kw)
        check(3)
    for i, fraction in ((0, 0.0), (1, 0.06)):
        nx, ny = SIZES[i]
        for sim in pairs[i]:
            sim.set_geometry(inputs.random_solid_mask(nx, ny, seed=40 + i, fraction=fraction))
            sim.init_fields(*inputs.random_fields(nx, ny, 50 + i, umax=0.05))
    check(5)
    batch.close()
