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
