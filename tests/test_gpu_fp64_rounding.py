"""Rounding of the FP64 step: no further from the exact step than a plain
double evaluation of Eqs. 1-5 that takes one direction at a time."""
import numpy as np
import pytest

from paper_2009_12584_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a GPU", allow_module_level=True)

from paper_2009_12584_gb300 import lbm  # noqa: E402

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)


def _step(f, tau, G, T):
    """One step of a fully periodic box without solids in the precision T:
    f_i(x, t) [2][9][ny][nx] to f_i(x, t + 1)."""
    f = f.astype(T)
    w = [T(4) / T(9)] + [T(1) / T(9)] * 4 + [T(1) / T(36)] * 4
    at = lambda q, i: np.roll(q, (-CY[i], -CX[i]), (0, 1))  # q(x + c_i)
    rho = [((p[0] + (p[1] + p[3])) + (p[2] + p[4])) + ((p[5] + p[7]) + (p[6] + p[8])) for p in f]
    F = [[-rho[s] * (T(G) * sum(w[i] * c[i] * at(rho[1 - s], i) for i in range(1, 9))) for c in (CX, CY)]
         for s in range(2)]
    j = [sum(c[i] * f[s][i] for s in range(2) for i in range(1, 9)) for c in (CX, CY)]
    u = [(j[d] + T(0.5) * (F[0][d] + F[1][d])) / (rho[0] + rho[1]) for d in range(2)]
    usq = T(1.5) * (u[0] * u[0] + u[1] * u[1])
    out = np.empty_like(f)
    for s in range(2):
        om, kF = T(1) / T(tau[s]), T(1) - T(1) / (T(2) * T(tau[s]))
        gain = T(0)
        for i in range(1, 9):
            cu, cF = CX[i] * u[0] + CY[i] * u[1], CX[i] * F[s][0] + CY[i] * F[s][1]
            S = w[i] * kF * ((T(3) * cF - T(3) * (u[0] * F[s][0] + u[1] * F[s][1])) + T(9) * cu * cF)
            r = w[i] * rho[s]
            d = om * ((r - f[s][i]) + r * (cu * (T(3) + T(4.5) * cu) - usq)) + S
            gain = gain + d
            out[s][i] = np.roll(f[s][i] + d, (CY[i], CX[i]), (0, 1))
        out[s][0] = f[s][0] - gain
    return out


@pytest.mark.parametrize("kernel", ["two_pass", "tiled", "halo", "fused"])
@pytest.mark.parametrize("tau", [(0.6, 0.6), (0.8, 1.3), (1.6, 1.6)])
def test_fp64_step_rounds_like_the_plain_form(kernel, tau):
    """rms over the 16 moving populations of 96 x 64 nodes, some steps after a
    rough start: their errors are a few independent roundings each, so the rms
    of 98,304 of them is known to 0.3%; 5% are allowed."""
    nx, ny = 96, 64
    sim = lbm.Simulation(nx, ny, storage="fp64", kernel=kernel, periodic_x=True, periodic_y=True, tau=tau)
    sim.set_geometry(np.zeros((ny, nx), np.uint8)).set_wetting("martys_chen")
    sim.init_fields(*inputs.random_fields(nx, ny, 4, umax=0.05)).step(20)
    f = sim.populations().cpu().numpy()
    got = sim.step(1).populations().cpu().numpy()
    exact = _step(f, tau, 3.0, np.longdouble)
    plain = _step(f, tau, 3.0, np.float64)
    rms = lambda a: float(np.sqrt(np.mean((a[:, 1:].astype(np.longdouble) - exact[:, 1:]) ** 2)))
    assert rms(got) < 1.05 * rms(plain)
    assert rms(plain) < 1e-16  # the reference forms agree
