"""Served requests of mixed sizes: small batches beside batches that fill the GPU (sent in
slices), in numbers on both sides of the rule for sharing the SMs, against plain runs."""
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


@pytest.mark.parametrize("batches", [(20_011, 12_000_000, 11_000_003), (20_011, 12_000_000, 30_000, 9_001, 11_000_003)])
def test_mixed_requests_equal_plain_runs(ctd, batches):
    p = [I.head(1, seed=90 + i, shape=(18, 20, 14 + i), d=1.1) for i in range(len(batches))]
    c = ctd.ctd_create(device=0, serve_round_histories=1e9)
    hs = [ctd.load_problem(c, x) for x in p]
    ids = [ctd.ctd_submit(c, h, B, 0.0, x.seed, n_histories_max=(2 + i) * B, min_batches=2)
           for i, (h, x, B) in enumerate(zip(hs, p, batches))]
    for i in ids:
        assert ctd.ctd_wait(c, i, 60.0)["state"] == ctd.REQ_DONE
    plain = ctd.ctd_create(device=0)
    for i, (h, x, B) in enumerate(zip(hs, p, batches)):
        dose, sd, st = ctd.ctd_get_dose_and_stddev(c, h, x.phantom.nvox)
        d1, s1, t1, _ = ctd.run_problem(plain, I.scaled(x, n_hist=(2 + i) * B, n_batches=2 + i))
        assert [st[q] for q in COUNTS] == [t1[q] for q in COUNTS]
        assert np.allclose(dose, d1, rtol=1e-12, atol=0)
    ctd.ctd_destroy(plain)
    ctd.ctd_destroy(c)
