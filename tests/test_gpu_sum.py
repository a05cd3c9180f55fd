"""The FP64 concentration (a sum of nine populations taken in integers) over
populations of every scale, sign and spread: each fluid node's C after one
step of a closed box, against exact rational sums of what it pulls.

The sum is off by half an ulp of itself and at most 9/64 ulp of its largest
term, so |C - exact| <= 2^-53 |exact| + 9 * 2^-58 * max |g|, the bound used
(2^-52 and 2^-54 of them).  Terms beyond the integer path (the largest below
2^-943 or from 2^1016, infinite, NaN) are added in order, as by numpy."""
import struct

from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
NX, NY = 32, 8


def _states():
    rng = np.random.RandomState(3)
    shape = (9, NY, NX)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    plain = w * (1 + 0.2 * rng.standard_normal(shape))
    yield "plain", plain
    yield "signs", plain * rng.choice([-1.0, 1.0], shape)
    yield "spread", plain * 10.0 ** rng.uniform(-25, 25, shape)
    yield "dilute", plain * 10.0 ** rng.uniform(-250, -200, (1, NY, NX))
    yield "cancel", np.where(np.arange(9)[:, None, None] % 2 == 0, 1.0,
                             -1.0) * (1 + 1e-13 * rng.standard_normal(shape))
    yield "zeros", np.where(rng.random_sample(shape) < 0.7, 0.0, plain)
    yield "tiny", plain * 10.0 ** rng.uniform(-320, -280, (1, NY, NX))
    yield "huge", plain * 10.0 ** rng.uniform(300, 307, (1, NY, NX))
    bad = plain.copy()
    bad[3, 2, 5], bad[4, 5, 20] = np.inf, np.nan
    yield "infinite", bad


@pytest.mark.parametrize("name,g", list(_states()), ids=lambda v: v if
                         isinstance(v, str) else "")
def test_concentration_sum(name, g):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    geom = lbm.Geometry(NX, NY, np.zeros((0, 6)), 0.0, 0.0)
    geom.set_periodic(lbm.LBM_PERIODIC_X | lbm.LBM_PERIODIC_Y).upload()
    u = torch.zeros((2, NY, NX), dtype=torch.float64, device="cuda")
    # C after two steps sums what the second one pulls, the populations that
    # the first one (of a solver of its own) left
    prm = lbm.adr_params(1, 1e300, precision=lbm.LBM_F64, neg_tol=-1.0)
    first, sv = (lbm.ADRSolver(geom, prm, u).init() for _ in range(2))
    buf = sv.state_save()
    head = buf.size - 9 * NX * NY * 8
    assert struct.unpack_from("<q", buf.tobytes(), 32)[0] == 0   # steps
    buf[head:] = np.frombuffer(np.ascontiguousarray(g).tobytes(), np.uint8)
    first.state_load(buf).run(1, check=False)
    sv.state_load(buf)
    if name == "infinite":
        with pytest.raises(lbm.LBMError):
            sv.run(2)
    else:
        sv.run(2)
    got = sv.conc().cpu().numpy()[0]
    moved = first.state_save()[head:].view(np.float64).reshape(9, NY, NX)
    pulled = np.stack([np.roll(moved[i], (CY[i], CX[i]), (0, 1))
                       for i in range(9)])
    in_order = pulled[0].copy()
    with np.errstate(over="ignore", invalid="ignore"):
        for i in range(1, 9):
            in_order = in_order + pulled[i]
    largest = np.abs(pulled).max(0)
    beyond = ~((largest == 0) | ((largest >= 2.0 ** -943) &
                                 (largest < 2.0 ** 1016)))
    assert beyond.any() or name not in ("tiny", "huge", "infinite")
    assert np.array_equal(got[beyond], in_order[beyond], equal_nan=True)
    for y, x in zip(*np.nonzero(~beyond)):
        p = pulled[:, y, x]
        exact = sum(Fraction(float(v)) for v in p)
        bound = Fraction(2) ** -52 * abs(exact) + \
            Fraction(2) ** -54 * Fraction(float(largest[y, x]))
        assert abs(Fraction(float(got[y, x])) - exact) <= bound
