"""A batched call after its phantom was destroyed and created again.  The context hands
released device buffers out again first in, first out by their size, so the new phantom
can have every buffer of the old one but its densities; the recorded batch may not be
replayed then, for its statistics kernels would read the old densities.  Here a dense
phantom becomes one whose every other voxel is below the measures' 0.1 g/cm^3."""
import numpy as np
import pytest

from paper_1109_3266_gb300 import inputs as I

pytestmark = pytest.mark.gpu

N, NB = 40_000, 4


@pytest.fixture(scope="module")
def ctd():
    from paper_1109_3266_gb300 import build, ctd as binding
    build.build()
    return binding


def problem(thin):
    ph = I.uniform_box(20, 18, 16, 0.6)
    rho = np.ones_like(ph.rho)
    if thin:
        rho.reshape(-1)[::2] = 0.05
    return I.Problem("replay", I.Phantom(20, 18, 16, 0.6, 0.6, 0.6, ph.mat, rho, ph.materials),
                     I.arc_source(100.0, -4.0, 4.0, -3.0, 3.0, n_proj=90), I.spectrum_kramers(100, 2.5), I.Physics(),
                     N, NB, 17)


# (three spare blocks of the densities' size: the second phantom after the recorded one
# gets the recorded one's buffers but for the densities; without them, all of them)
@pytest.mark.parametrize("spare", [0, 1, 2, 3, 4])
def test_recreated_phantom_is_measured_by_its_own_densities(ctd, spare):
    c = ctd.ctd_create(device=0)
    # phantoms of four times the voxels: their material arrays have the size of the densities
    p0 = problem(False)
    big = I.uniform_box(40, 36, 16, 0.3)
    others = [ctd.ctd_create_phantom(c, 40, 36, 16, 0.3, 0.3, 0.3, big.mat, big.rho, big.materials) for _ in range(spare)]
    for step, thin in enumerate((False, True, True)):
        p = problem(thin)
        h = ctd.load_problem(c, p)
        if step != 1:   # recorded by the first phantom; the second takes its buffers in turn
            ctd.ctd_run_batch(c, [h], [N], [p.seed], NB)
        else:
            ctd.ctd_run(c, h, N, p.seed, NB)
        dose, sd, st = ctd.ctd_get_dose_and_stddev(c, h, p0.phantom.nvox)
        mask = p.phantom.rho.reshape(-1) >= np.float32(0.1)
        dmax = dose[mask].max()
        m1, m2 = mask & (dose > 0.1 * dmax), mask & (dose > 0.2 * dmax)
        assert st["d_max"] == dmax
        assert st["avg_rsd"] == pytest.approx((sd[m1] / dose[m1]).mean(), rel=1e-12)
        assert st["paper_sigma_bar"] == pytest.approx(sd[m2].mean() / dmax, rel=1e-12)
        for o in others:
            ctd.ctd_destroy_phantom(c, o)
        others = []
        ctd.ctd_destroy_phantom(c, h)
    ctd.ctd_destroy(c)
