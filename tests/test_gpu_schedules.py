"""Choices the step makes by size and state: launch shapes, and what one
wetting scheme leaves in the workspace for the next."""
import numpy as np
import pytest

from paper_2009_12584_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2009_12584_gb300 import lbm  # noqa: E402

IMPROVED = ("virtual_avg", dict(G_s=(3.0, 3.0), chi=(1.2, 0.8)))
SCHEMES = {
    "mc": ("martys_chen", dict(G_s=(-0.2, 0.2))),
    "llkc": ("llkc", dict(G_s=(-0.5, 0.3), pairing=lbm.PAIR_SELF)),
    "constant": ("constant", dict(G_s=(3.0, 2.5), rho_s=(0.3, 0.7))),
}


def _sim(nx, ny, storage, kernel, wet, mask, seed=5):
    sim = lbm.Simulation(nx, ny, storage=storage, kernel=kernel, periodic_x=True, periodic_y=True)
    sim.set_geometry(mask).set_wetting(wet[0], **wet[1])
    rA, rB, ux, uy = inputs.random_fields(nx, ny, seed, umax=0.05)
    return sim.init_fields(rA, rB, ux, uy)


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("kernel", ["auto", "two_pass", "tiled"])
@pytest.mark.parametrize("scheme", sorted(SCHEMES))
def test_scheme_after_improved_starts_clean(storage, kernel, scheme):
    """Steps after a change from the improved scheme equal those of a
    context that never ran it (its solid cells hold no virtual densities)."""
    nx, ny = 70, 45
    mask = inputs.random_solid_mask(nx, ny, seed=3, fraction=0.25)
    a = _sim(nx, ny, storage, kernel, IMPROVED, mask)
    a.step(6)
    f = a.populations()
    b = _sim(nx, ny, storage, kernel, SCHEMES[scheme], mask)
    a.set_populations(f)
    b.set_populations(f)
    a.set_wetting(SCHEMES[scheme][0], **SCHEMES[scheme][1])
    assert torch.equal(a.forces(), b.forces())
    a.step(5)
    b.step(5)
    assert torch.equal(a.populations(), b.populations())


@pytest.mark.parametrize("nx,ny", [(61, 40), (333, 121), (800, 510)])
def test_fp64_auto_matches_tiled(nx, ny):
    """AUTO's FP64 step (one-warp CTAs, then 128 threads above 16 CTAs per
    SM) and the tiled step give the same bits."""
    mask = inputs.random_solid_mask(nx, ny, seed=7, fraction=0.05)
    a, b = (_sim(nx, ny, "fp64", k, IMPROVED, mask) for k in ("auto", "tiled"))
    a.step(4)
    b.step(4)
    assert torch.equal(a.populations(), b.populations())
    assert np.all(np.isfinite(a.mass()))


# Tile edges of the halo schedule: 32 columns, 14 rows (20 with 16-bit
# storage), one tile, one node more, a ragged last tile, windows that reach
# across a whole small periodic box.
@pytest.mark.parametrize("storage,vref", [("fp32", False), ("fp64", False), ("fp16", False), ("bf16", False),
                                          ("fp16", True), ("bf16", True)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (32, 14), (33, 15), (32, 20), (65, 41), (100, 61), (31, 13)])
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("scheme", ["improved", "improved_d2q9_self", "llkc", "constant"])
def test_halo_matches_two_pass_bitwise(storage, vref, nx, ny, periodic, scheme):
    wet = {"improved": IMPROVED,
           "improved_d2q9_self": ("virtual_avg", dict(G_s=(2.5, 3.5), chi=(0.9, 1.3), pairing=lbm.PAIR_SELF,
                                                      avg_stencil=9))}.get(scheme) or SCHEMES[scheme]
    mask = inputs.random_solid_mask(nx, ny, seed=nx + ny, fraction=0.12, periodic_x=periodic, periodic_y=periodic)
    rA, rB, ux, uy = inputs.random_fields(nx, ny, 11, umax=0.05)
    out = []
    for kernel in ("two_pass", "halo"):
        sim = lbm.Simulation(nx, ny, storage=storage, velocity_refs=vref, kernel=kernel, periodic_x=periodic,
                             periodic_y=periodic)
        sim.set_geometry(mask).set_wetting(wet[0], **wet[1]).init_fields(rA, rB, ux, uy)
        sim.step(3)
        m = sim.moments()  # in the middle: the next steps start from the same state
        sim.step(4)
        sim.sync()
        out.append([*m, sim.populations(), torch.from_numpy(sim.mass())])
        sim.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)


def test_halo_without_room_for_its_lists_runs_two_pass():
    """A workspace with a small interface list leaves no room for the lists
    of a 16-bit context: the same results, by the two-pass schedule."""
    nx, ny = 96, 70
    mask = inputs.flat_wall_mask(nx, ny)
    rA, rB, ux, uy = inputs.random_fields(nx, ny, 2, umax=0.05)
    out = []
    for cap in (0, 2 * nx):
        sim = lbm.Simulation(nx, ny, storage="fp16", kernel="halo", periodic_x=True, max_interface=cap)
        sim.set_geometry(mask).set_wetting(IMPROVED[0], **IMPROVED[1]).init_fields(rA, rB, ux, uy)
        n0 = sim.launch_count
        sim.step(5)
        out.append((sim.launch_count - n0, sim.populations()))
        sim.close()
    assert out[0][0] == 5 and out[1][0] == 15  # one launch a step; density, Eq. 8, collide
    assert torch.equal(out[0][1], out[1][1])


def test_halo_wait_runs_out_and_context_recovers():
    """A tile whose copies do not complete within the bound is reported, later
    steps do nothing until then, and the context steps on afterwards."""
    nx, ny = 70, 50
    mask = inputs.inclined_wall_mask(nx, ny, 20.0, 9)
    rA, rB = inputs.sharp_droplet(nx, ny, nx / 2, ny / 2, 9)
    sims = []
    for kernel in ("halo", "two_pass"):
        sim = lbm.Simulation(nx, ny, kernel=kernel)
        sims.append(sim.set_geometry(mask).set_wetting(IMPROVED[0], **IMPROVED[1]).init_fields(rA, rB))
    sims[0].step(2).debug_tma_expect_extra(16)
    sims[0].step(3)
    with pytest.raises(lbm.LbmError) as e:
        sims[0].sync()
    assert e.value.status == lbm.ERR_TIMEOUT
    sims[0].debug_tma_expect_extra(0).sync()
    sims[0].init_fields(rA, rB).step(7)
    sims[1].step(7)
    sims[0].sync()
    assert torch.equal(sims[0].populations(), sims[1].populations())


@pytest.mark.parametrize("storage", ["fp32", "fp64", "fp16", "bf16"])
@pytest.mark.parametrize("graph", [0, 2])
def test_batch_of_mixed_members_matches_members_alone(storage, graph):
    """One batch over everything its list schedule tells apart: one ring and
    three, with and without velocity references, members of the two passes
    among those of the halo kernel, sizes below and above a tile; odd step
    counts, and a member that starts from the other buffer."""
    kinds = [(4, 4, "auto", IMPROVED, False), (33, 21, "two_pass", IMPROVED, False),
             (70, 45, "auto", SCHEMES["llkc"], False), (64, 40, "halo", IMPROVED, True),
             (32, 14, "auto", SCHEMES["mc"], True), (100, 61, "two_pass", SCHEMES["constant"], True)]
    pairs = []
    for i, (nx, ny, kernel, wet, vref) in enumerate(kinds):
        two = []
        for _ in range(2):
            sim = lbm.Simulation(nx, ny, storage=storage, kernel=kernel, periodic_x=True, periodic_y=True,
                                 velocity_refs=vref and storage in ("fp16", "bf16"))
            sim.set_geometry(inputs.random_solid_mask(nx, ny, seed=i, fraction=0.1)).set_wetting(wet[0], **wet[1])
            rA, rB, ux, uy = inputs.random_fields(nx, ny, 20 + i, umax=0.05)
            two.append(sim.init_fields(rA, rB, ux, uy).step(i % 2))
        pairs.append(two)
    batch = lbm.Batch([p[0] for p in pairs])
    if graph:
        batch.set_graph_steps(graph)
    for n in (1, 4, 3):
        batch.step(n)
        for a, b in pairs:
            b.step(n)
            a.sync()
            assert torch.equal(a.populations(), b.populations())
    for a, b in pairs:  # and alone again
        assert torch.equal(a.step(2).populations(), b.step(2).populations())
    batch.close()


@pytest.mark.parametrize("storage,vref", [("fp32", False), ("fp16", False), ("bf16", True)])
@pytest.mark.parametrize("scheme", ["improved", "llkc"])
def test_moments_of_halo_contexts_match_the_general_evaluation(storage, vref, scheme):
    """The halo kernel's moments against the density, Eq. 8 and evaluation
    passes of a two-pass context, on a ragged grid; each array may be left
    out or lie on any byte."""
    nx, ny = 75, 43
    wet = IMPROVED if scheme == "improved" else SCHEMES[scheme]
    mask = inputs.random_solid_mask(nx, ny, seed=4, fraction=0.15, periodic_x=True, periodic_y=False)
    rA, rB, ux, uy = inputs.random_fields(nx, ny, 6, umax=0.05)
    sims = []
    for kernel in ("auto", "two_pass"):
        sim = lbm.Simulation(nx, ny, storage=storage, velocity_refs=vref, kernel=kernel, periodic_x=True)
        sim.set_geometry(mask).set_wetting(wet[0], **wet[1]).init_fields(rA, rB, ux, uy)
        sims.append(sim.step(3))
    a, b = (torch.cat([m.reshape(-1) for m in s.moments()]) for s in sims)
    assert torch.equal(a, b)
    n = nx * ny * 8
    raw = torch.full((n + 16,), 7, dtype=torch.uint8, device="cuda")
    for off, field in ((0, 2), (3, 1)):
        ptr = [None] * 4
        ptr[field] = raw.data_ptr() + off
        assert sims[0].lib.lbm_moments(sims[0].h, *ptr) == lbm.OK
        got = raw[off:off + n].clone().view(torch.float64)
        assert torch.equal(got, a[field * nx * ny:(field + 1) * nx * ny])
        assert torch.all(raw[off + n:] == 7)


@pytest.mark.parametrize("nx,ny", [(8, 8), (300, 200), (512, 300)])
def test_diagnostics_at_block_edges(nx, ny):
    """Fewer blocks than the reduction's 256, about one node per thread, and
    several, with a bridge longer than the 32 rows of one scan: against the
    same sums of the moments."""
    mask = np.zeros((ny, nx), np.uint8)
    rA = np.full((ny, nx), 0.05)
    rA[: ny * 2 // 3, : nx * 2 // 3] = 1.0
    sim = lbm.Simulation(nx, ny, storage="fp64", kernel="two_pass", periodic_x=True, periodic_y=True)
    sim.set_geometry(mask).set_wetting("martys_chen").init_fields(rA, 1.05 - rA, np.full((ny, nx), 0.01),
                                                                 np.zeros((ny, nx)))
    r, _, u = (m.cpu().numpy() for m in sim.moments())
    d = sim.diagnostics(level=0.5, rho_out=0.055, bridge=(1, 1), wall_point=(0.0, -100.0))
    w = np.maximum(r - 0.055, 0.0)
    yy, xx = np.mgrid[0:ny, 0:nx]
    assert abs(d["weight"] - w.sum()) < 1e-9 * w.sum()
    assert abs(d["com"][0] - (w * xx).sum() / w.sum()) < 1e-9 * nx
    assert abs(d["com"][1] - (w * yy).sum() / w.sum()) < 1e-9 * ny
    assert abs(d["max_u"] - np.sqrt((u ** 2).sum(0).max())) < 1e-12
    above = r >= 0.5
    cross = (above[:, :-1] != above[:, 1:]).sum() + (above[:-1] != above[1:]).sum()
    assert d["contour_points"] == cross and d["nonfinite_nodes"] == 0
    y1 = ny * 2 // 3  # the first row below the level
    t = (r[y1 - 1, 1] - 0.5) / (r[y1 - 1, 1] - r[y1, 1])
    assert abs(d["bridge_radius"] - (y1 - 1 + t - 0.5)) < 1e-9
