"""Two FP32 steps per launch on lattices that take them although their last
strip of 254 columns is in part idle: the state is the same bits as that of
single steps, over link types, flags and edges, and so is what a checked run
after them reports (both forms round every operation alike)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_04455_gb300 import _build
    _build.build()


def _solvers(nx, ny, ns, flags, periodic):
    assert lbm.load().lbm_adr_steps_per_launch(lbm.LBM_F32, ns, nx, ny) == 2
    rng = np.random.RandomState(nx)
    rows = [[rng.uniform(0, nx), rng.uniform(0, ny), rng.uniform(2, 30), k % 4,
             rng.uniform(0, 6), -1 if k % 5 else 0.4] for k in range(150)]
    # fibers across the lattice's edges and the last strip's
    rows += [[x, y, 9.0, 1 + i % 3, 0.5, -1] for i, (x, y) in enumerate(
        [(0, 0), (nx - 1, ny // 2), (nx // 2, ny - 1),
         ((nx - 1) // 254 * 254 - 0.5, 31.5)])]
    geom = lbm.Geometry(nx, ny, np.array(rows), 0.3, 0.2)
    if periodic:
        geom.set_periodic(periodic)
    geom.upload()
    gen = torch.Generator(device="cuda").manual_seed(nx)
    u = 0.06 * (torch.rand((2, ny, geom.nx_pad), generator=gen,
                           device="cuda") - 0.5)
    prm = lbm.adr_params(ns, [0.6, 0.8, 1.1], c_in=(1.0, 0.3, 0.2),
                         precision=lbm.LBM_F32, flags=flags, neg_tol=-1.0)
    return geom, [lbm.ADRSolver(geom, prm, u).init() for _ in range(2)]


@pytest.mark.parametrize("nx,ny,ns,flags,periodic", [
    (2287, 2700, 3, 0, 3), (4573, 2000, 2, lbm.LBM_ADR_INLET_ABB_ALL, 0),
    (601, 14001, 3, lbm.LBM_ADR_NODEWISE, 2), (140001, 32, 2, 0, 1)])
def test_two_steps_equal_single_steps(nx, ny, ns, flags, periodic):
    _, (a, b) = _solvers(nx, ny, ns, flags, periodic)
    a.run(5, check=False)
    for _ in range(5):
        b.run(1, check=False)
    assert np.array_equal(a.state_save(), b.state_save())
    # four plain steps, two at a time and one by one, then two checked ones
    got = a.run(6)
    for _ in range(4):
        b.run(1, check=False)
    assert got == b.run(2)
    assert np.array_equal(a.state_save(), b.state_save())


def test_two_steps_follow_a_new_upload():
    """Edges made periodic and uploaded into the same workspace hold for a
    solver that was created before."""
    geom, (a, b) = _solvers(4573, 2000, 2, 0, 0)
    ws = geom.ws.data_ptr()
    for flags in (0, 3, 1, 2, 0):
        geom.set_periodic(flags)
        geom.upload()
        assert geom.ws.data_ptr() == ws
        a.run(4, check=False)
        for _ in range(4):
            b.run(1, check=False)
        assert np.array_equal(a.state_save(), b.state_save())
