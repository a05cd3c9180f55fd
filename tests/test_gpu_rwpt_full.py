"""A full particle buffer: the particles in the box keep their places and only
entrance particles are dropped, however the two kinds are appended.

Particles at rest, none of which leaves but those of the entrance strip, in a
buffer that the initial fill takes up to the last slot; a seed for which more
particles enter than the strip had held."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rwpt as orwpt  # noqa: E402
from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu

NX, NY, DENSITY = 60, 40, 20.0
ENTER = int(DENSITY * NY)


def _fill():
    fib = np.array([[12.0 + 6 * i, 8.0 + 12 * j, 1.5, 0, 0, -1]
                    for i in range(8) for j in range(3)])
    for seed in range(100):
        kw = dict(D=0.0, density=DENSITY, radius_offset=0.5, seed=seed, nspecies=2)
        r = orwpt.RWPT(NX, NY, fib, 0.0, 0.0, None, **kw).init()
        x, y, _, ids = r.p.sorted()
        if ENTER - int((x < 0.5).sum()) >= 20:
            return fib, kw, x, y, ids
    raise AssertionError("no such seed")


@pytest.mark.parametrize("room", [0, 10, 20 * ENTER])
def test_particles_in_the_box_come_first(room):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fib, kw, x, y, ids = _fill()
    stay = x >= 0.5
    capacity = len(ids) + room
    g = lbm.RWPT(NX, NY, fib, 0.0, 0.0, None, capacity=capacity, **kw).init()
    for step in range(100):
        g.run(1, report=False)
        gx, gy, gs, gid = g.particles()
        old = gid < int(DENSITY * NX * NY)
        assert np.array_equal(gid[old], ids[stay])
        assert np.array_equal(gx[old], x[stay]) and np.array_equal(gy[old], y[stay])
        # the strip holds entrance particles of this step alone
        first = int(DENSITY * NX * NY) + step * ENTER
        new = gid[~old]
        assert np.all((new >= first) & (new < first + ENTER))
        assert len(gid) == min(capacity, int(stay.sum()) + ENTER)
    if room <= 10:
        with pytest.raises(lbm.LBMError) as e:
            g.run(1)
        assert e.value.status == lbm.LBM_ENOMEM
    else:
        assert g.run(1)["overflow"] == 0
