"""A batched call whose batches share launches in groups with a shorter last one, on
scratch that chains of one stream use one after another, against a launch per batch."""
import numpy as np
import pytest

from paper_1109_3266_gb300 import inputs as I

pytestmark = pytest.mark.gpu

COUNTS = ("pe", "compton", "rayleigh", "fictitious", "escaped", "missed", "cutoff", "terminated", "aborted", "steps")


@pytest.fixture(scope="module")
def ctd():
    from paper_1109_3266_gb300 import build, ctd as binding
    build.build()
    return binding


# 128 tallies of 128^3 voxels fill half of the scratch: groups of 128 and 2, and of 128,
# 128 and 3, for two requests on two streams, which two small ones share
@pytest.mark.parametrize("nb", [130, 259])
def test_groups_with_a_shorter_last_one(ctd, nb):
    ps = [I.cbct_water(50_021, nb, seed=3, shape=(128, 128, 128), d=0.2), I.head(40_000, nb, seed=4, shape=(128, 128, 128), d=0.2),
          I.head(9_001, nb, seed=5, shape=(20, 18, 16), d=1.0), I.cbct_water(7_000, nb, seed=6, shape=(33, 20, 9), d=0.8)]
    c, plain = ctd.ctd_create(device=0), ctd.ctd_create(device=0, plain_overlap=1)
    hs = [ctd.load_problem(c, p) for p in ps]
    for _ in range(2):   # recorded, then replayed on the tallies the folds left cleared
        ctd.ctd_run_batch(c, hs, [p.n_hist for p in ps], [p.seed for p in ps], nb)
        got = [ctd.ctd_get_dose_and_stddev(c, h, p.phantom.nvox) for h, p in zip(hs, ps)]
    ctd.ctd_destroy(c)
    for p, (dose, sd, st) in zip(ps, got):
        d1, s1, t1, h = ctd.run_problem(plain, p)
        ctd.ctd_destroy_phantom(plain, h)
        assert [st[k] for k in COUNTS] == [t1[k] for k in COUNTS]
        assert np.allclose(dose, d1, rtol=1e-12, atol=0)
        # a variance is a difference of sums: its rounding is relative to the squared mean
        assert np.allclose(sd ** 2, s1 ** 2, rtol=1e-9, atol=1e-12 * float((d1 ** 2).max()))
        assert st["e_deposited_kev"] == pytest.approx(t1["e_deposited_kev"], rel=1e-12)
    ctd.ctd_destroy(plain)
