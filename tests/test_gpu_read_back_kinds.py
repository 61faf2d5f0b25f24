"""Reading grids back into pinned and managed memory, beside an output in new plain
memory whose pages threads make: the same values as in a buffer in use."""
import ctypes as C

import numpy as np
import pytest

from paper_1109_3266_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctd():
    from paper_1109_3266_gb300 import build, ctd as binding
    build.build()
    return binding


@pytest.mark.parametrize("kind", ["pinned", "managed"])
@pytest.mark.parametrize("first", [False, True])
def test_destinations_that_cuda_knows(ctd, kind, first):
    import torch

    n = 1_048_577
    ph = I.Phantom(n, 1, 1, 20.0 / n, 5.0, 5.0, np.zeros((1, 1, n), np.uint8), np.ones((1, 1, n), np.float32), [I.WATER])
    p = I.Problem("strip", ph, I.static_source(50.0, 8.0, 2.0), I.spectrum_line(60.0), I.Physics(), 20_000, 2, 3)
    ctx = ctd.ctd_create(device=0)
    h = ctd.load_problem(ctx, p)
    ctd.ctd_run(ctx, h, p.n_hist, p.seed, p.n_batches)
    ref = [np.full(n, -7.0) for _ in range(2)]
    dp = C.POINTER(C.c_double)
    assert ctd.lib().ctd_get_dose_and_stddev(ctx, h, *(a.ctypes.data_as(dp) for a in ref), n, None) == 0
    torch.zeros(1, device="cuda")
    rt, ptr = C.CDLL("libcudart.so.13"), C.c_void_p()   # the one torch has loaded
    if kind == "pinned":
        assert rt.cudaMallocHost(C.byref(ptr), C.c_size_t(8 * n)) == 0
    else:
        assert rt.cudaMallocManaged(C.byref(ptr), C.c_size_t(8 * n), C.c_uint(1)) == 0
    known = np.ctypeslib.as_array(C.cast(ptr, dp), (n,))
    new = np.empty(n)
    out = (known, new) if first else (new, known)
    assert ctd.lib().ctd_get_dose_and_stddev(ctx, h, *(a.ctypes.data_as(dp) for a in out), n, None) == 0
    assert np.array_equal(out[0], ref[0]) and np.array_equal(out[1], ref[1])
    assert (rt.cudaFreeHost if kind == "pinned" else rt.cudaFree)(ptr) == 0
    ctd.ctd_destroy(ctx)
    assert ref[0].max() > 0.0
