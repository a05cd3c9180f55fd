"""The particle read-back in the order of the ids (a radix sort of the free
buffer on the device): the same particles as the CPU oracle's, bit for bit,
at counts around a sort tile (2048) and a digit of the ids (256, 65536), with
the smallest capacities (below 293 the host sorts) and with a full buffer."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import rwpt as orwpt  # noqa: E402
from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,spare", [
    (1, 0), (1, 400), (40, 252), (40, 253), (256, 300), (257, 5), (2047, 0),
    (2048, 0), (2049, 1), (4097, 0), (66000, 7)])
def test_particles_come_in_id_order(count, spare):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # a periodic box of `count` particles: none enters or leaves
    nx = ny = 16
    kw = dict(D=0.3, dt=0.5, delta=0.2, density=count / (nx * ny),
              radius_offset=0.0, seed=count, nspecies=2)
    fib = np.zeros((0, 6))
    g = lbm.RWPT(nx, ny, fib, 0.2, 0.0, None, capacity=count + spare,
                 flags=lbm.LBM_RWPT_PERIODIC | lbm.LBM_RWPT_HOMOGENEOUS,
                 **kw).init()
    r = orwpt.RWPT(nx, ny, fib, 0.2, 0.0, None, periodic=True,
                   homogeneous=True, **kw).init()
    for n in (0, 3, 2):   # the sort's scratch is the next step's buffer
        if n:
            g.run(n)
            r.run(n)
        got, want = g.particles(), r.p.sorted()
        ids = got[3]
        assert len(ids) == count and np.all(ids[1:] > ids[:-1])
        for a, b in zip((got[3], got[2], got[0], got[1]),
                        (want[3], want[2], want[0], want[1])):
            assert np.array_equal(a, b)
