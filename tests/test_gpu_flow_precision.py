"""The FP64 flow against the same scheme in extended precision (numpy's
longdouble: 64 bits of mantissa on x86, 113 on Arm).

What leads the error of a double run is a systematic loss of mass: weights
rounded to double add up to 1 - 6e-17, so that plain formulas lose that part
of the density times 1/tau per step, 3e-14 to 6e-14 of the velocities in 400
steps of this lattice.  A step whose constants conserve mass exactly is left
with roundings that do not add up: 9 populations of at most 0.45 rounded to
2^-55 of it each and some ten operations before that, in quadrature over 400
steps 20 * 2^-53 * 4 = 9e-15 of the density 1, of which the velocity, 0.05 and
driven by differences of the density, sees a part.  The bound is 2e-14."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu

NX, NY, STEPS, U0 = 48, 24, 400, 0.05
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
L = np.longdouble
W = [L(4) / 9] + [L(1) / 9] * 4 + [L(1) / 36] * 4


def _velocity_after(solid, tau, steps):
    """u after `steps` pull steps from the parabolic start."""
    y = np.arange(NY).astype(L)[:, None]
    u_in = 4 * L(U0) * (y + L(0.5)) * (NY - L(0.5) - y) / (L(NY) * NY)
    fluid = ~solid

    def equilibrium(i, rho, ux, uy):
        cu, uu = CX[i] * ux + CY[i] * uy, ux * ux + uy * uy
        return W[i] * rho * (1 + 3 * cu + L(4.5) * cu * cu - L(1.5) * uu)

    ux, uy = np.where(fluid, u_in, L(0)), np.zeros((NY, NX), L)
    f = [np.where(fluid, equilibrium(i, L(1), ux, uy), L(0)) for i in range(9)]
    padded = np.pad(solid, 1, constant_values=True)   # walls above and below
    for _ in range(steps):
        rho = sum(f)
        ux = sum(CX[i] * f[i] for i in range(9)) / np.where(fluid, rho, 1)
        uy = sum(CY[i] * f[i] for i in range(9)) / np.where(fluid, rho, 1)
        post = [f[i] + (equilibrium(i, rho, ux, uy) - f[i]) / L(tau)
                for i in range(9)]
        wx, wy = (sum(c[i] * post[i][:, -1] for i in range(9)) /
                  sum(p[:, -1] for p in post) for c in (CX, CY))
        new = []
        for i in range(9):
            dy, dx = CY[i], CX[i]
            pulled = np.roll(post[i], (dy, dx), (0, 1))
            source = padded[1 - dy:1 - dy + NY, 1 - dx:1 - dx + NX]
            g = np.where(source, post[OPP[i]], pulled)
            if dx == 1:     # from beyond the inlet
                g[:, 0] = (post[OPP[i]] + 6 * W[i] * u_in)[:, 0]
            elif dx == -1:  # from beyond the outlet
                cu, uu = dx * wx + dy * wy, wx * wx + wy * wy
                g[:, -1] = (2 * W[i] * (1 + L(4.5) * cu * cu - L(1.5) * uu) -
                            post[OPP[i]][:, -1])
            new.append(np.where(fluid, g, L(0)))
        f = new
    rho = np.where(fluid, sum(f), 1)
    return np.stack([sum(c[i] * f[i] for i in range(9)) / rho for c in (CX, CY)])


@pytest.mark.parametrize("tau", [0.56, 0.8, 1.3])
def test_flow_keeps_its_mass(tau):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yy, xx = np.mgrid[0:NY, 0:NX]
    fiber = (0.4 * NX, 0.5 * NY, NY / 10.0)
    solid = (xx - fiber[0]) ** 2 + (yy - fiber[1]) ** 2 <= fiber[2] ** 2
    geom = lbm.Geometry(NX, NY, np.array([[*fiber, 0, 0, -1]]), 0.0, 0.0).upload()
    u, _ = lbm.lbm_flow_solve(geom, tau, U0, STEPS, precision=lbm.LBM_F64)
    got = u.cpu().numpy()[:, :, :NX].astype(L)
    want = _velocity_after(solid, tau, STEPS)
    assert np.sum((got - want) ** 2) <= L(2e-14) ** 2 * np.sum(want ** 2)
