"""Particles that a velocity field carries to NaN, of either sign, or to an
infinity leave through the outlet and are counted, as in the CPU oracle
(not x < nx - 1/2); the others go on unchanged."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rwpt as orwpt  # noqa: E402
from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.filterwarnings("ignore::RuntimeWarning")
@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf],
                         ids=["nan", "negative nan", "infinity"])
def test_particles_without_a_position_leave(bad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny = 48, 24
    fib = np.array([[12.0, 12.0, 4.0, 3, 0.3, -1], [36.0, 6.0, 3.0, 1, 0, -1]])
    ux, uy = np.full((ny, nx), 0.15), np.zeros((ny, nx))
    ux[:, 24:28] = bad   # every particle that comes by, of any species
    uy[3:6, 8] = bad if np.isnan(bad) else 0.0   # out a step later, by x
    assert np.signbit(ux[0, 24]) == np.signbit(bad)
    u = torch.zeros((2, ny, (nx + 31) // 32 * 32), dtype=torch.float64)
    u[0, :, :nx], u[1, :, :nx] = torch.from_numpy(ux), torch.from_numpy(uy)
    kw = dict(D=0.2, dt=0.5, delta=0.5, density=6.0, radius_offset=0.5, seed=4,
              nspecies=3)
    g = lbm.RWPT(nx, ny, fib, 0.5, 0.4, u.cuda(), capacity=20000, **kw).init()
    r = orwpt.RWPT(nx, ny, fib, 0.5, 0.4, (ux, uy), **kw).init()
    for n in (1, 5, 60):
        info = g.run(n)
        r.run(n)
        assert list(info["out"]) == list(r.out)
        got, want = g.particles(), r.p.sorted()
        assert info["alive"] == len(want[3])
        for a, b in zip(got, want):
            assert np.array_equal(a, b, equal_nan=a.dtype.kind == "f")
    assert (r.out[:2] > 0).all()
