"""How many steps the library takes per launch, as it tells and as the
benchmark's record counts launches and bytes (host arithmetic, no GPU)."""
import types

import pytest

import bench
from paper_2109_04455_gb300 import lbm


@pytest.fixture(scope="module")
def steps():
    from paper_2109_04455_gb300 import _build
    _build.build()
    return lbm.load().lbm_adr_steps_per_launch


def test_limits(steps):
    for prec in (lbm.LBM_F64, lbm.LBM_F32, lbm.LBM_F16DEV):
        for ns in (1, 2, 3):
            two = prec == lbm.LBM_F32 and ns >= 2
            assert steps(prec, ns, 16384, 4096) == (2 if two else 1)
            assert steps(prec, ns, 2048, 1024) == 1
            assert steps(prec, ns, 4, 1) == 1
    # the kernel's 32-bit population numbers: 9 ns plane < 2^32
    assert steps(lbm.LBM_F32, 3, 65536, 2427) == 2
    assert steps(lbm.LBM_F32, 3, 65536, 2428) == 1
    assert steps(lbm.LBM_F32, 2, 65536, 2428) == 2
    assert steps(lbm.LBM_F32, 2, 65536, 3641) == 1
    # (the largest lattices: no overflow on the way)
    assert steps(lbm.LBM_F32, 3, 2**31 - 1, 65535) == 1


def test_arguments_no_solver_takes(steps):
    ok = [lbm.LBM_F32, 3, 4096, 4096]
    for k, bad in ((0, -1), (0, 3), (1, 0), (1, 4), (2, 3), (3, 0), (3, 65536)):
        args = list(ok)
        args[k] = bad
        assert steps(*args) == 0


@pytest.mark.parametrize("nx,ny,two,three", [
    # steps per launch with two and three species: whole strips of 254 columns,
    # or lattices so large or flat that a strip in part idle does not matter
    (4096, 2048, 2, 2), (16384, 1024, 2, 2), (140000, 32, 2, 2),
    (1 << 20, 4, 2, 2), (2048, 8192, 2, 2),
    # two species move less, and so gain less
    (2032, 2100, 1, 2), (4096, 1100, 1, 2), (1020, 16000, 1, 2), (600, 14000, 1, 2),
    # strips much of which is idle: single steps are faster
    (2048, 2048, 1, 1), (1020, 4200, 1, 1), (1280, 3300, 1, 1), (510, 8300, 1, 1),
    (430, 10000, 1, 1), (260, 16384, 1, 1), (256, 16500, 1, 1), (300, 14500, 1, 1),
    (160, 27000, 1, 1)])
def test_strip_fill(steps, nx, ny, two, three):
    assert (nx + 31) // 32 * 32 * ny >= 1 << 22
    assert steps(lbm.LBM_F32, 2, nx, ny) == two
    assert steps(lbm.LBM_F32, 3, nx, ny) == three


@pytest.mark.parametrize("precision", ["f64", "f32", "f16dev"])
@pytest.mark.parametrize("nx,ny", [(2048, 512), (16384, 4096), (65536, 4096)])
def test_benchmark_counts_what_the_library_does(steps, precision, nx, ny):
    geom = types.SimpleNamespace(nx=nx, ny=ny, nx_pad=(nx + 31) // 32 * 32)
    prec = {"f64": lbm.LBM_F64, "f32": lbm.LBM_F32, "f16dev": lbm.LBM_F16DEV}
    assert bench._steps_per_launch(geom, precision) == \
        steps(prec[precision], bench.SPECIES, nx, ny)
