"""The bounded wait of the halo step's copies, made to run out on the host's
word (the barriers expect more bytes than the copies deliver, so no wait can
complete; nothing faults): what each caller hears, and what the CTAs that had
not started yet do."""
import time

import pytest

from paper_2009_12584_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2009_12584_gb300 import lbm  # noqa: E402

WET = dict(G_s=(3.0, 3.0), chi=(1.2, 0.8))


def _sim(nx, ny, storage="fp32", kernel="auto", vref=False):
    mask = inputs.inclined_wall_mask(nx, ny, 20.0, 9)
    sim = lbm.Simulation(nx, ny, storage=storage, kernel=kernel, velocity_refs=vref)
    sim.set_geometry(mask).set_wetting("virtual_avg", **WET)
    return sim.init_fields(*inputs.sharp_droplet(nx, ny, nx / 2, ny / 2, 9))


def _times_out(call):
    with pytest.raises(lbm.LbmError) as e:
        call()
    assert e.value.status == lbm.ERR_TIMEOUT


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_wait_runs_out_in_a_grid_of_several_waves(storage):
    """More tiles than the chip holds at once: the CTAs of the later waves find
    the error word set by the first, while others of their wave may still be
    setting it, and end as a whole; so do the moments of that state. The
    waits run out once, not once per wave, and the context steps on."""
    nx, ny = 1504, 1000
    sim = _sim(nx, ny, storage).step(1)
    sim.sync()
    sim.debug_tma_expect_extra(16)
    t0 = time.time()
    sim.step(2).moments()
    _times_out(sim.sync)
    assert 0.5 < time.time() - t0 < 10.0
    sim.debug_tma_expect_extra(0).sync()
    rA, rB = inputs.sharp_droplet(nx, ny, nx / 2, ny / 2, 9)
    ref = _sim(nx, ny, storage, "two_pass")
    assert torch.equal(sim.init_fields(rA, rB).step(3).populations(), ref.step(3).populations())
    sim.sync()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("call", ["diagnostics", "mass", "set_geometry", "run_host", "run_host_f32", "step_profiled"])
def test_every_synchronising_call_reports_the_timeout(call, storage):
    """What waits for a step's results says that there are none, once, and the
    next use of the context is sound again."""
    nx, ny = 70, 50
    sim = _sim(nx, ny, storage).step(2)
    before = sim.diagnostics()
    mask = sim.mask.cpu().numpy()
    rA, rB = inputs.sharp_droplet(nx, ny, nx / 2, ny / 2, 9)
    wet = lbm.make_wetting("virtual_avg", **WET)

    def run_host():
        import numpy as np
        t = np.float64 if call == "run_host" else np.float32
        out = [np.empty((ny, nx), t) for _ in range(4)]
        getattr(sim, call)(wet, mask, rA.astype(t), rB.astype(t), 2, out)
        return out

    calls = dict(diagnostics=sim.diagnostics, mass=sim.mass, set_geometry=lambda: sim.set_geometry(mask),
                 step_profiled=lambda: sim.step_profiled(1), run_host=run_host, run_host_f32=run_host)
    sim.debug_tma_expect_extra(16)
    if not call.startswith("run_host"):
        sim.step(1)
        moments = sim.moments()
        _fluid = torch.from_numpy(mask == 0).cuda()
        for m in (moments[0], moments[1], moments[2][0], moments[2][1]):
            assert torch.all(torch.isnan(m[_fluid])) and torch.all(m[~_fluid] == 0)
    _times_out(calls[call])
    sim.debug_tma_expect_extra(0).sync()
    sim.set_geometry(mask).init_fields(rA, rB).step(2)
    assert sim.diagnostics() == before
    if call.startswith("run_host"):
        assert torch.equal(torch.from_numpy(run_host()[0]).cuda(), sim.moments()[0].to(
            torch.float64 if call == "run_host" else torch.float32))


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("graph", [0, 2])
def test_batch_tells_every_member_that_missed_a_step(storage, graph):
    """One member's wait runs out: the halo members, of both launches, miss the
    steps that follow and all say so, the one of the two passes does not; the
    batch refuses to step on from there until they have said it."""
    sizes = [(70, 50, "auto", "virtual_avg"), (96, 61, "auto", "virtual_avg"), (130, 70, "halo", "llkc"),
             (64, 40, "two_pass", "virtual_avg")]

    def member(nx, ny, kernel, scheme):
        sim = _sim(nx, ny, storage, kernel)
        return sim.set_wetting(scheme, **(WET if scheme == "virtual_avg" else dict(G_s=(-0.5, 0.3))))

    sims = [member(*z) for z in sizes]
    batch = lbm.Batch(sims)
    if graph:
        batch.set_graph_steps(graph)
    batch.step(1)
    sims[1].debug_tma_expect_extra(16)
    batch.step(4)
    sims[1].debug_tma_expect_extra(0)
    _times_out(lambda: batch.step(1))
    for sim in sims[:2]:
        _times_out(sim.sync)
    _times_out(lambda: batch.step(1))
    _times_out(sims[2].sync)
    for sim in sims:
        sim.sync()
    for sim, z in zip(sims, sizes):
        sim.init_fields(*inputs.sharp_droplet(z[0], z[1], z[0] / 2, z[1] / 2, 9))
    batch.step(5)
    for sim, z in zip(sims, sizes):
        sim.sync()
        assert torch.equal(sim.populations(), member(*z).step(5).populations())
    batch.close()
