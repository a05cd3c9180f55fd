"""Reading the particles (which sorts them in the buffer of the next step)
beside other work on the same system: on another stream than the steps, which
are still running, and from several threads at once.  Every read gives the
particles of a system that ran alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2109_04455_gb300 import lbm  # noqa: E402

pytestmark = pytest.mark.gpu

STEPS = 300


def _system():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    fib = np.array([[40.0 + 30 * i, 20.0 + 25 * j, 6.0, 1 + (i + j) % 3, 0.4, -1]
                    for i in range(6) for j in range(4)])
    return lbm.RWPT(256, 110, fib, 0.3, 0.2, None, D=0.2, density=8.0, seed=3,
                    nspecies=3, capacity=400000)


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


def test_read_on_another_stream():
    alone, g = _system(), _system()
    steps, reads = torch.cuda.Stream(), torch.cuda.Stream()
    alone.init()
    torch.cuda.synchronize()
    g.init(stream=steps)
    for _ in range(3):
        alone.run(STEPS)
        g.run(STEPS, stream=steps, report=False)
        got = g.particles(stream=reads)   # the steps are still under way
        assert _same(got, alone.particles())


def test_reads_from_several_threads():
    g = _system().init()
    g.run(STEPS)
    want = g.particles()
    bad = []

    def read(stream):
        with torch.cuda.stream(stream):
            for _ in range(10):
                if not _same(g.particles(), want):
                    bad.append(stream)

    threads = [threading.Thread(target=read, args=(torch.cuda.Stream(),))
               for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    g.run(STEPS)   # and the system goes on as if it had not been read
    alone = _system().init()
    alone.run(2 * STEPS)
    assert _same(g.particles(), alone.particles())
