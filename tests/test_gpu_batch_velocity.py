"""A batch takes each lattice's velocity wherever its first value lies: a view
into a larger buffer, one, two or three values past a 16-byte boundary, gives
the same bits as an aligned copy in every precision (half storage loads two
and four velocities at a time).  A pointer between two values is refused."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [(130, 40), (65, 33), (257, 24)]   # rows past a tile, ragged ends


@pytest.fixture(scope="module")
def geoms():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_04455_gb300 import _build
    _build.build()
    return [lbm.Geometry(nx, ny, np.array([[0.4 * nx, 0.5 * ny, 5.0, 3, 0.4, -1],
                                           [0.7 * nx, 0.2 * ny, 4.0, 1, 0, -1]]),
                         0.3, 0.2).upload() for nx, ny in SHAPES]


def _at(value, offset):
    """A copy of `value` whose first element lies `offset` elements past a
    256-byte boundary."""
    buf = torch.empty(value.numel() + 64, dtype=value.dtype, device="cuda")
    start = (-buf.data_ptr() // value.element_size()) % (256 // value.element_size())
    out = buf[start + offset:start + offset + value.numel()].view(value.shape)
    out.copy_(value)
    assert out.data_ptr() % 256 == offset * value.element_size()
    return out


@pytest.mark.parametrize("prec", [lbm.LBM_F64, lbm.LBM_F32, lbm.LBM_F16DEV])
def test_velocity_views(geoms, prec):
    gen = torch.Generator(device="cuda").manual_seed(5)
    us = [(0.1 * torch.rand((2, g.ny, g.nx_pad), generator=gen, device="cuda",
                            dtype=torch.float64) - 0.05) for g in geoms]
    if prec != lbm.LBM_F64:
        us = [u.float() for u in us]
    params = [lbm.adr_params(3, 0.8, precision=prec, max_steps=20, check_every=10,
                             neg_tol=-1.0) for _ in geoms]
    want = None
    for offset in (0, 1, 2, 3):
        b = lbm.Batch(geoms, params, [_at(u, offset) for u in us])
        # (the other sums' order follows the launch shape, which is timed)
        got = [[i["steps"], i["flux"], b.conc(k).cpu().numpy()]
               for k, i in enumerate(b.solve())]
        if want is None:
            want = got
        for g, w in zip(got, want):
            assert g[:2] == w[:2] and np.array_equal(g[2], w[2])


@pytest.mark.parametrize("prec", [lbm.LBM_F64, lbm.LBM_F32, lbm.LBM_F16DEV])
def test_velocity_between_values_is_refused(geoms, prec):
    class Odd:   # never read: the call that binds it is refused
        def __init__(self, u):
            self.u = u

        def data_ptr(self):
            return self.u.data_ptr() + self.u.element_size() // 2

    dtype = torch.float64 if prec == lbm.LBM_F64 else torch.float32
    us = [torch.zeros((2, g.ny, g.nx_pad), dtype=dtype, device="cuda") for g in geoms]
    params = [lbm.adr_params(3, 0.8, precision=prec, max_steps=20) for _ in geoms]
    with pytest.raises(lbm.LBMError) as e:
        lbm.Batch(geoms, params, us[:2] + [Odd(us[2])])
    assert e.value.status == lbm.LBM_EINVAL
