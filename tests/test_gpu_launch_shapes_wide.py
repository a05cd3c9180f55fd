"""Every precision of the lattice kernels at the edges of their launch shapes,
against the FP64 CPU oracle: 64-thread segments (a node short of, at and past
one), and 256-thread segments with a partial last one.

256 threads are taken from four 256-node segments per SM for the FP64 ADR step
(608 of them) and from sixteen for the flow and the FP32 step (2432), where
they cover at most a quarter more than the row: 470 columns are two segments
of a padded row of 480.  (Of the shapes in test_gpu_launch_shapes.py 250 x 620
alone takes 256-thread segments, one whole one per row, in the FP64 ADR step;
513 x 620, whose padding is too wide, and all flows there take 64 threads.)
Half storage covers 256-node segments at any size, four nodes per thread on
plain steps and two on checked ones.

Bounds.  40 steps of about 10 roundings of a unit u each per population, in a
map that amplifies nothing: 40 * 10 * u, for double 4.5e-14 (bound 1e-12) and
float 2.4e-5.  Half storage rounds the deviation from the node's concentration,
below a quarter of a population at the sharpest front, by at most 2^-10 of it,
up or down at random: 40 steps add up to 40^0.5 * 2^-12 = 1.6e-3 of the
population where the front is, and no more of the norm.  One node in error
alone, by as much as the flux of one link, a 36th, shows in the largest
difference: bound 1e-2 of the inlet concentration."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu

STEPS = 40
NARROW = [(63, 9), (64, 24), (65, 24), (129, 40), (257, 130), (259, 33)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_04455_gb300 import _build
    _build.build()
    oracle.build()


def _lattice(nx, ny):
    r = min(nx, ny) / 8.0
    fib = np.array([[0.30 * nx, 0.30 * ny, r, 1, 0, -1],
                    [0.55 * nx, 0.65 * ny, r, 2, 0, -1],
                    [0.80 * nx, 0.35 * ny, r, 3, 0.7, -1],
                    [0.30 * nx, 0.75 * ny, 0.6 * r, 0, 0, -1],
                    [254.0, 0.5 * ny, 3.0, 1, 0, 0.4]])   # across a segment's end
    return fib, oracle.raster(nx, ny, fib, 0.2, 0.3)


@pytest.mark.parametrize("prec,shape", [
    *((p, s) for p in (lbm.LBM_F32, lbm.LBM_F16DEV) for s in NARROW),
    (lbm.LBM_F64, (470, 310)), (lbm.LBM_F32, (470, 1220)),
    (lbm.LBM_F16DEV, (470, 310))])
@pytest.mark.parametrize("ns", [1, 2, 3])
def test_adr_step(prec, shape, ns):
    nx, ny = shape
    fib, (solid, kab, kbc) = _lattice(nx, ny)
    y = (np.arange(ny) + 0.5) / ny
    ux = np.where(solid, 0.0, (0.2 * y * (1 - y))[:, None] * np.ones(nx))
    uy = np.where(solid, 0.0, 0.01 * np.sin(np.arange(nx) / 9.0)[None, :] *
                  np.ones((ny, 1)))
    taus, cin = [0.6, 0.75, 0.9][:ns], [1.0, 0.0, 0.0][:ns]
    geom = lbm.Geometry(nx, ny, fib, 0.2, 0.3).upload()
    u = torch.zeros((2, ny, geom.nx_pad),
                    dtype=torch.float64 if prec == lbm.LBM_F64 else torch.float32)
    u[0, :, :nx], u[1, :, :nx] = torch.from_numpy(ux), torch.from_numpy(uy)
    prm = lbm.adr_params(ns, taus, precision=prec, max_steps=STEPS, neg_tol=-1.0)
    conc, _ = lbm.lbm_adr_solve(geom, prm, u.cuda())
    ref = oracle.ADRProblem(solid, kab, kbc, ux, uy, taus, cin).run(STEPS)
    got = conc.cpu().numpy()[:, :, :nx].astype(np.float64)
    rel, most = {lbm.LBM_F64: (1e-12, 1e-12), lbm.LBM_F32: (2.4e-5, 2.4e-5),
                 lbm.LBM_F16DEV: (1.6e-3, 1e-2)}[prec]
    for s in range(ns):
        d = got[s] - ref["conc"][s]
        # (a species that barely exists yet: relative to all of them)
        assert np.linalg.norm(d) <= rel * np.linalg.norm(ref["conc"])
        assert np.abs(d).max() <= most


@pytest.mark.parametrize("prec", [lbm.LBM_F64, lbm.LBM_F32])
def test_flow_step_of_256_threads(prec):
    nx, ny = 470, 1220
    fib, (solid, _, _) = _lattice(nx, ny)
    geom = lbm.Geometry(nx, ny, fib, 0.2, 0.3).upload()
    u, info = lbm.lbm_flow_solve(geom, 0.7, 0.05, STEPS, precision=prec)
    _, ux, uy, res = oracle.flow_run(solid, 0.7, 0.05, STEPS)
    got = u.cpu().numpy()[:, :, :nx].astype(np.float64)
    # velocities are differences of populations of order one: 40 steps of
    # about 20 roundings of 1.1e-16 (6e-8) each
    bound = 1e-13 if prec == lbm.LBM_F64 else 5e-5
    assert np.abs(got[0] - ux).max() < bound
    assert np.abs(got[1] - uy).max() < bound
    if prec == lbm.LBM_F64:
        assert info["residual"] == pytest.approx(res, rel=1e-8)
