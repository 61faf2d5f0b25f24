"""Reading grids back into pages that do not exist yet, made by several threads a
chunk at a time, against reading them into a buffer in use: at the sizes where the
threads start (4 MiB of outputs) and where chunks end (8 MiB), at addresses off a
page's start, with the memory around the outputs left alone."""
import ctypes as C
import mmap

import numpy as np
import pytest

from paper_1109_3266_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctd():
    from paper_1109_3266_gb300 import build, ctd as binding
    build.build()
    return binding


@pytest.mark.parametrize("n", [1, 262_143, 262_144, 524_289, 1_048_575, 1_048_576, 1_048_577, 4_000_003])
def test_cold_and_warm_destinations(ctd, n):
    ph = I.Phantom(n, 1, 1, 20.0 / n, 5.0, 5.0, np.zeros((1, 1, n), np.uint8), np.ones((1, 1, n), np.float32), [I.WATER])
    p = I.Problem("strip", ph, I.static_source(50.0, 8.0, 2.0), I.spectrum_line(60.0), I.Physics(), 20_000, 2, 3)
    ctx = ctd.ctd_create(device=0)
    h = ctd.load_problem(ctx, p)
    ctd.ctd_run(ctx, h, p.n_hist, p.seed, p.n_batches)
    warm = [np.full(n + 2, -7.0) for _ in range(3)]   # a guard on either side
    f = lambda a: a[1:].ctypes.data_as(C.POINTER(C.c_double))
    assert ctd.lib().ctd_get_dose_and_stddev(ctx, h, f(warm[0]), f(warm[1]), n, None) == 0
    assert ctd.lib().ctd_get_edep(ctx, h, f(warm[2]), n) == 0
    bytes_ = 8 * (n + 2)
    maps = [mmap.mmap(-1, bytes_ + 4096) for _ in range(3)]
    cold = [np.frombuffer(m, dtype=np.float64, count=n + 2, offset=40) for m in maps]   # pages untouched so far
    assert ctd.lib().ctd_get_dose_and_stddev(ctx, h, f(cold[0]), f(cold[1]), n, None) == 0
    assert ctd.lib().ctd_get_edep(ctx, h, f(cold[2]), n) == 0
    ctd.ctd_destroy(ctx)
    for w, c in zip(warm, cold):
        assert w[0] == -7.0 and w[-1] == -7.0 and c[0] == 0.0 and c[-1] == 0.0
        assert np.array_equal(w[1:-1], c[1:-1])
    assert warm[0][1:-1].max() > 0.0 and warm[2][1:-1].sum() > 0.0
