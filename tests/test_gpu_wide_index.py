"""Phantoms at the limit of the fast index arithmetic: a voxel index comes from
positions truncated by an addition of 2^23, which holds for axes of up to 2^23
voxels; longer axes take the instantiation with conversion instructions.  Both
sides of the line against the binary64 oracle, history by history.  The water is
uniform, so that a voxel boundary decides nothing but the deposit's place, which
may be off by binary32's resolution in voxel units: eps = 2^-24 times 16 (SAD +
half diagonal) / d for the entry point, 26 n for the moved position, and 64 free
paths / d (the bounds the decision margins use for one flight)."""
import numpy as np
import pytest

from paper_1109_3266_gb300 import inputs as I
from track_compare import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctd():
    from paper_1109_3266_gb300 import build, ctd as binding
    build.build()
    return binding


@pytest.mark.parametrize("axis", [0, 2])
@pytest.mark.parametrize("n", [2 ** 23, 2 ** 23 + 1])
def test_long_axis_history_by_history(ctd, oracle, axis, n):
    dims = [1, 1, 1]
    dims[axis] = n
    size = [10.0, 10.0, 10.0]
    size[axis] = 10.0 / n
    nx, ny, nz = dims
    ph = I.Phantom(nx, ny, nz, *size, np.zeros((nz, ny, nx), np.uint8), np.ones((nz, ny, nx), np.float32), [I.WATER])
    p = I.Problem("long_axis", ph, I.static_source(50.0, 4.0, 4.0), I.spectrum_line(60.0),
                  I.Physics(mode="max_real", max_real=1), 20_000, 2, 7)
    ctx = ctd.ctd_create(device=0)
    h = ctd.load_problem(ctx, p)
    dev = ctd.ctd_trace_range(ctx, h, p.n_hist, p.seed, p.n_batches, 0, p.n_hist)
    ctd.ctd_run(ctx, h, p.n_hist, p.seed, p.n_batches)   # the production instantiation
    _, _, st = ctd.ctd_get_dose_and_stddev(ctx, h, ph.nvox, want_arrays=False)
    ctd.ctd_destroy(ctx)
    ref = oracle.Setup(p, 64).track(0, p.n_hist, threads=16)
    s = compare(dev, ref)
    assert s["never_ended"] == 0 and s["mismatches"] <= 5e-3 * p.n_hist, s
    free_path = 5.5   # cm of water at 60 keV, rounded up
    bound = 2.0 ** -24 * ((16 * (50.0 + 8.7) + 64 * free_path) / size[axis] + 26 * n)
    same = (dev["end"] == ref["end"]) & (dev["last_type"] >= 0)
    off = np.abs(dev["idx"][same].astype(np.int64) - ref["idx"][same].astype(np.int64))
    assert off.max() <= bound, (off.max(), bound)
    assert st["steps"] == int(dev["steps"].sum()) and st["pe"] == int((dev["end"] == 0).sum())
