"""Two FP32 steps per launch (lattices of at least 2^22 nodes): the state is
the same bits as that of single steps, over every link type, flag and edge,
at widths around a whole number of the kernel's 254-column strips.

Both forms round every operation of a node's update alike, so nothing is
allowed to differ.  run(1) never takes two steps at once."""
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
    lbm.load()


def _fibers(nx, ny):
    rng = np.random.RandomState(nx)
    rows = [[rng.uniform(0, nx), rng.uniform(0, ny), rng.uniform(2, 40),
             k % 4, rng.uniform(0, 6), -1 if k % 5 else 0.4]
            for k in range(150)]
    # fibers across the edges of the lattice and of strips and runs of rows
    rows += [[x, y, 9.0, 1 + (i % 3), 0.5, -1] for i, (x, y) in enumerate(
        [(0, 0), (nx - 1, ny // 2), (nx // 2, ny - 1), (253.5, 31.5),
         (254, 64), (508, 0)])]
    return np.array(rows)


@pytest.mark.parametrize("nx,ny,ns,flags,periodic", [
    (2032, 2080, 3, 0, 0), (2033, 2101, 3, 0, 3), (2031, 2077, 2, 0, 1),
    (4099, 1040, 3, lbm.LBM_ADR_NODEWISE, 2),
    (140000, 32, 3, lbm.LBM_ADR_INLET_ABB_ALL, 0),
    (256, 16500, 2, lbm.LBM_ADR_NODEWISE | lbm.LBM_ADR_INLET_ABB_ALL, 0)])
def test_two_steps_equal_single_steps(nx, ny, ns, flags, periodic):
    geom = lbm.Geometry(nx, ny, _fibers(nx, ny), 0.3, 0.2)
    if periodic:
        geom.set_periodic(periodic)
    geom.upload()
    assert geom.nx_pad * ny >= 1 << 22
    gen = torch.Generator(device="cuda").manual_seed(nx)
    u = 0.06 * (torch.rand((2, ny, geom.nx_pad), generator=gen,
                           device="cuda") - 0.5)
    prm = lbm.adr_params(ns, [0.6, 0.8, 1.1], c_in=(1.0, 0.3, 0.2),
                         precision=lbm.LBM_F32, flags=flags, neg_tol=-1.0)
    a = lbm.ADRSolver(geom, prm, u).init()
    b = lbm.ADRSolver(geom, prm, u).init()
    for n in (7, 2):
        a.run(n, check=False)
        for _ in range(n):
            b.run(1, check=False)
    assert np.array_equal(a.state_save(), b.state_save())
    # and so is what a checked run reports
    assert a.run(6) == b.run(6)


def test_two_steps_follow_a_new_upload():
    """Edges made periodic and uploaded into the same workspace hold for a
    solver that was created before, as they do for single steps."""
    nx, ny = 2033, 2101
    geom = lbm.Geometry(nx, ny, _fibers(nx, ny), 0.3, 0.2)
    geom.upload()
    u = torch.zeros((2, ny, geom.nx_pad), device="cuda")
    u[:, :, :nx] = 0.03
    prm = lbm.adr_params(2, [0.6, 0.8], c_in=(1.0, 0.3), precision=lbm.LBM_F32,
                         neg_tol=-1.0)
    a = lbm.ADRSolver(geom, prm, u).init()
    b = lbm.ADRSolver(geom, prm, u).init()
    ws = geom.ws.data_ptr()
    for flags in (0, 3, 1, 2, 0):
        geom.set_periodic(flags)
        geom.upload()
        assert geom.ws.data_ptr() == ws
        a.run(4, check=False)
        for _ in range(4):
            b.run(1, check=False)
        assert np.array_equal(a.state_save(), b.state_save())
