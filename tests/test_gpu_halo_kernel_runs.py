"""The halo kernel against the two passes where it is certain that it ran: one
launch per step, in contexts with room for its lists (a large max_interface),
so that 16-bit storage takes part on every grid, periodic ones included."""
import pytest

from paper_2009_12584_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2009_12584_gb300 import lbm  # noqa: E402

SCHEMES = {
    "improved": ("virtual_avg", dict(G_s=(3.0, 3.0), chi=(1.2, 0.8))),
    "improved_d2q9_self": ("virtual_avg", dict(G_s=(2.5, 3.5), chi=(0.9, 1.3), pairing=lbm.PAIR_SELF, avg_stencil=9)),
    "llkc": ("llkc", dict(G_s=(-0.5, 0.3), pairing=lbm.PAIR_SELF)),
}
STORAGE = [("fp32", False), ("fp64", False), ("fp16", False), ("bf16", False), ("fp16", True), ("bf16", True)]


def _sim(nx, ny, storage, vref, kernel, scheme, periodic, seed, fraction=0.12):
    mask = inputs.random_solid_mask(nx, ny, seed=seed, fraction=fraction, periodic_x=periodic, periodic_y=periodic)
    sim = lbm.Simulation(nx, ny, storage=storage, velocity_refs=vref, kernel=kernel, periodic_x=periodic,
                         periodic_y=periodic, max_interface=8 * nx * ny + 4096)
    sim.set_geometry(mask).set_wetting(SCHEMES[scheme][0], **SCHEMES[scheme][1])
    return sim.init_fields(*inputs.random_fields(nx, ny, seed + 1, umax=0.05))


# Tiles of 32 x 16 nodes (4- and 8-byte storage) and 32 x 20 (16-bit): one
# tile, one node less and more, two, ragged last tiles, and boxes so small that
# a window wraps around them.
@pytest.mark.parametrize("storage,vref", STORAGE)
@pytest.mark.parametrize("nx,ny", [(4, 4), (31, 15), (32, 16), (33, 17), (32, 20), (33, 21), (31, 19), (64, 32), (64, 40),
                                   (100, 61)])
@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("scheme", sorted(SCHEMES))
def test_one_launch_per_step_and_the_bits_of_two_passes(storage, vref, nx, ny, periodic, scheme):
    a, b = (_sim(nx, ny, storage, vref, k, scheme, periodic, nx + ny) for k in ("halo", "two_pass"))
    fluid = bool((a.mask == 0).any())
    n0 = a.launch_count
    a.step(3)
    assert a.launch_count - n0 == (3 if fluid else 0)
    n0 = a.launch_count
    m = a.moments()
    if fluid and storage != "fp64":
        assert a.launch_count - n0 == 2  # moments, zeros at solid nodes
    for x, y in zip(m, b.step(3).moments()):
        assert torch.equal(x, y)
    assert torch.equal(a.step(4).populations(), b.step(4).populations())
    assert torch.equal(torch.from_numpy(a.mass()), torch.from_numpy(b.mass()))


@pytest.mark.parametrize("storage", ["fp16", "bf16", "fp32"])
@pytest.mark.parametrize("graph", [0, 2])
def test_every_batched_halo_launch(storage, graph):
    """Members of one ring and of three, with and without velocity references
    (16-bit storage): a launch per kind and step, and the bits of each alone."""
    kinds = [(75, 45, "improved", False), (33, 21, "llkc", False), (64, 40, "improved_d2q9_self", True),
             (100, 61, "llkc", True), (32, 20, "improved", True), (4, 4, "improved", False)]
    make = lambda i, k: _sim(k[0], k[1], storage, k[3] and storage != "fp32", "auto", k[2], True, 3 + i, 0.1)
    pairs = [[make(i, k) for _ in range(2)] for i, k in enumerate(kinds)]
    pairs[0][0].step(1), pairs[0][1].step(1)  # one member starts from the other buffer
    batch = lbm.Batch([p[0] for p in pairs])
    batch.set_graph_steps(graph)
    for n in (1, 4, 3):
        n0 = batch.launch_count
        batch.step(n)
        assert batch.launch_count - n0 == n * (2 if storage == "fp32" else 4)
        for a, b in pairs:
            a.sync()
            assert torch.equal(a.populations(), b.step(n).populations())
            for x, y in zip(a.moments(), b.moments()):
                assert torch.equal(x, y)
    batch.close()
