"""Lattices at the edges of the step kernels' launch shapes (64- and
256-thread row segments, boundary chunks in further columns of blocks), with
every link type, against the FP64 CPU oracle.

FP64 on both sides differs by rounding order alone: 40 steps of a map that
amplifies nothing, about 10 roundings of 1.1e-16 each per step, leave a
relative difference below 40 * 10 * 1.1e-16 = 5e-14; the bound is 1e-12."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu

STEPS = 40
# one node short of, at and past a segment; more chunks than rows (a chunk
# column of its own per block); 256-thread segments (at least 608 of them,
# padding below a quarter)
# (250 x 620 alone takes the last, in the FP64 ADR step; the other 256-thread
# forms and the other precisions are in test_gpu_launch_shapes_wide.py)
SHAPES = [(63, 9), (64, 24), (65, 24), (129, 40), (24, 130), (250, 620),
          (513, 620)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_04455_gb300 import _build
    _build.build()
    oracle.build()
    lbm.load()


def _fibers(nx, ny):
    r = min(nx, ny) / 8.0
    return np.array([[0.30 * nx, 0.30 * ny, r, 1, 0, -1],
                     [0.55 * nx, 0.65 * ny, r, 2, 0, -1],
                     [0.80 * nx, 0.35 * ny, r, 3, 0.7, -1],
                     [0.30 * nx, 0.75 * ny, 0.6 * r, 0, 0, -1],
                     [0.78 * nx, 0.75 * ny, 0.6 * r, 1, 0, 0.4]])


def _velocity(nx, ny, solid):
    y = (np.arange(ny) + 0.5) / ny
    ux = np.where(solid, 0.0, (0.2 * y * (1 - y))[:, None] * np.ones(nx))
    uy = np.where(solid, 0.0, 0.01 * np.sin(np.arange(nx) / 9.0)[None, :] *
                  np.ones((ny, 1)))
    return ux, uy


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ns", [1, 2, 3])
def test_adr_step_shapes(shape, ns):
    nx, ny = shape
    fib = _fibers(nx, ny)
    solid, kab, kbc = oracle.raster(nx, ny, fib, 0.2, 0.3)
    ux, uy = _velocity(nx, ny, solid)
    taus, cin = [0.6, 0.75, 0.9][:ns], [1.0, 0.0, 0.0][:ns]
    geom = lbm.Geometry(nx, ny, fib, 0.2, 0.3).upload()
    u = torch.zeros((2, ny, geom.nx_pad), dtype=torch.float64)
    u[0, :, :nx], u[1, :, :nx] = torch.from_numpy(ux), torch.from_numpy(uy)
    prm = lbm.adr_params(ns, taus, precision=lbm.LBM_F64, max_steps=STEPS)
    conc, info = lbm.lbm_adr_solve(geom, prm, u.cuda())
    ref = oracle.ADRProblem(solid, kab, kbc, ux, uy, taus, cin).run(STEPS)
    got = conc.cpu().numpy()[:, :, :nx]
    for s in range(ns):
        assert np.linalg.norm(got[s] - ref["conc"][s]) <= \
            1e-12 * np.linalg.norm(ref["conc"][s])
    # the sums and the flux run over every row of the partials
    assert np.allclose(info["mass"][:ns], np.abs(ref["conc"]).sum((1, 2)),
                       rtol=1e-12, atol=0)
    assert np.allclose(info["flux"][:ns], ref["flux"][:ns], rtol=1e-10,
                       atol=1e-15)


@pytest.mark.parametrize("shape", SHAPES)
def test_flow_step_shapes(shape):
    nx, ny = shape
    fib = _fibers(nx, ny)
    solid, _, _ = oracle.raster(nx, ny, fib, 0.0, 0.0)
    geom = lbm.Geometry(nx, ny, fib, 0.0, 0.0).upload()
    u, info = lbm.lbm_flow_solve(geom, 0.7, 0.05, STEPS,
                                 precision=lbm.LBM_F64)
    _, ux, uy, res = oracle.flow_run(solid, 0.7, 0.05, STEPS)
    got = u.cpu().numpy()[:, :, :nx]
    # velocities are differences of populations of order one: 40 steps of
    # about 20 roundings of 1.1e-16 stay below 1e-13
    assert np.abs(got[0] - ux).max() < 1e-13
    assert np.abs(got[1] - uy).max() < 1e-13
    assert info["residual"] == pytest.approx(res, rel=1e-8)


@pytest.mark.parametrize("shape", [(65, 24), (250, 620)])
def test_flow_f32_keeps_its_density(shape):
    """The FP32 flow against the oracle after 400 steps: each step rounds to
    6e-8, with a systematic part below that (the weights as floats add up to
    1 - 3e-8), so the velocities stay within 400 * 6e-8 * 2 of 0.05 and
    relative; a density that drifts by another 1e-7 a step would not."""
    nx, ny = shape
    fib = _fibers(nx, ny)
    solid, _, _ = oracle.raster(nx, ny, fib, 0.0, 0.0)
    geom = lbm.Geometry(nx, ny, fib, 0.0, 0.0).upload()
    u, _ = lbm.lbm_flow_solve(geom, 0.8, 0.05, 400, precision=lbm.LBM_F32)
    _, ux, uy, _ = oracle.flow_run(solid, 0.8, 0.05, 400)
    got = u.cpu().numpy()[:, :, :nx].astype(np.float64)
    err = np.sqrt(np.sum((got[0] - ux) ** 2 + (got[1] - uy) ** 2))
    assert err <= 400 * 6e-8 * 2 * np.sqrt(np.sum(ux ** 2 + uy ** 2))
