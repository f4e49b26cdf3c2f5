"""lbm_moments into memory that a kernel of the context should not write."""
import numpy as np
import pytest

from paper_2009_12584_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2009_12584_gb300 import lbm  # noqa: E402


@pytest.mark.parametrize("storage,kernel", [("fp32", "auto"), ("fp64", "auto"), ("fp32", "two_pass")])
def test_moments_into_pinned_host_memory_are_copies(storage, kernel):
    """Fields in pinned host memory and on the device, mixed; the former come by
    way of the staging area, whose fields they leave there."""
    nx, ny = 70, 41
    sim = lbm.Simulation(nx, ny, storage=storage, kernel=kernel, periodic_x=True)
    sim.set_geometry(inputs.flat_wall_mask(nx, ny)).set_wetting("martys_chen", G_s=(-0.2, 0.2))
    sim.init_fields(*inputs.random_fields(nx, ny, 8, umax=0.05)).step(3)
    want = torch.cat([m.reshape(-1, ny, nx) for m in sim.moments()]).cpu()
    host = torch.full((4, ny, nx), -7.0, dtype=torch.float64).pin_memory()
    dev = torch.full((4, ny, nx), -7.0, dtype=torch.float64, device="cuda")
    assert sim.lib.lbm_moments(sim.h, host[0].data_ptr(), dev[1].data_ptr(), None, host[3].data_ptr()) == lbm.OK
    sim.sync()
    got = dev.cpu()
    for a, (h, d) in enumerate(((True, False), (False, True), (False, False), (True, False))):
        assert torch.equal(host[a], want[a]) if h else torch.all(host[a] == -7.0)
        assert torch.equal(got[a], want[a]) if d else torch.all(got[a] == -7.0)
    stage = sim.workspace.view(torch.uint8).cpu().numpy()
    for a in (0, 3):  # the fields that were copied are in the workspace too
        assert stage.tobytes().find(np.ascontiguousarray(want[a].numpy()).tobytes()) >= 0
