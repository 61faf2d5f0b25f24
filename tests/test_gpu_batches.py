"""Batches that share a transport launch (each with its own tally, folded in order)
against one launch per batch (the overlapped plain run), where the claims and the
batch boundaries meet: batches of one history, of just under and over a warp's
round, uneven batches, a launch with fewer histories than warps and one with more
than the small claims at its end cover.  Same histories, so the counts are equal;
deposits are binary32 numbers added in binary64, so the tallies differ by rounding
of at most n 2^-53 relative, far below 1e-12 here."""
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


@pytest.fixture(scope="module")
def contexts(ctd):
    cs = [ctd.ctd_create(device=0), ctd.ctd_create(device=0, plain_overlap=1)]
    yield cs
    for c in cs:
        ctd.ctd_destroy(c)


@pytest.mark.parametrize("n,nb", [(2, 2), (50, 50), (1_000, 37), (31 * 9 + 4, 9), (100_003, 7), (3_000_001, 5)])
def test_shared_launch_equals_launch_per_batch(ctd, contexts, n, nb):
    p = I.head(n, nb, seed=11, shape=(40, 37, 25), d=0.6)
    out = []
    for c in contexts:
        dose, sd, st, h = ctd.run_problem(c, p)
        edep = ctd.ctd_get_edep(c, h, p.phantom.nvox)
        ctd.ctd_destroy_phantom(c, h)
        out.append((dose, sd, edep, st))
    (d0, s0, e0, t0), (d1, s1, e1, t1) = out
    assert t0["transport_launches"] == 1 and t1["transport_launches"] == nb
    assert [t0[k] for k in COUNTS] == [t1[k] for k in COUNTS]
    assert sum(t0[k] for k in ("pe", "cutoff", "escaped", "missed", "terminated", "aborted")) == n
    assert t0["e_emitted_kev"] == t1["e_emitted_kev"] and t0["e_escaped_kev"] == t1["e_escaped_kev"]
    assert np.allclose(e0, e1, rtol=1e-12, atol=0) and np.allclose(d0, d1, rtol=1e-12, atol=0)
    # a variance is a difference of sums: its rounding is relative to the squared mean
    assert np.allclose(s0 ** 2, s1 ** 2, rtol=1e-9, atol=1e-12 * float((d0 ** 2).max()))


@pytest.mark.parametrize("n,nb,chunk", [(1_500_001, 4, 0), (2_801_665, 3, 0), (2_801_663, 3, 0), (9_000_011, 6, 0),
                                        (1_500_001, 4, 40), (5_000_000, 2, 1000)])
def test_claims_of_a_share_cover_every_history_once(ctd, contexts, n, nb, chunk):
    # claims of 32 to 256 histories by the launch's size (5472 warps: 32 and 64 meet at
    # 2801664), at most the option's; a launch per batch claims by each batch's size
    p = I.head(n, nb, seed=13, shape=(24, 22, 16), d=1.0)
    c = ctd.ctd_create(device=0, chunk=chunk)
    d0, s0, t0, h0 = ctd.run_problem(c, p)
    d1, s1, t1, h1 = ctd.run_problem(contexts[1], p)
    ctd.ctd_destroy_phantom(contexts[1], h1)
    ctd.ctd_destroy(c)
    assert [t0[k] for k in COUNTS] == [t1[k] for k in COUNTS]
    assert t0["e_emitted_kev"] == t1["e_emitted_kev"] and t0["e_escaped_kev"] == t1["e_escaped_kev"]
    assert np.allclose(d0, d1, rtol=1e-12, atol=0)


@pytest.mark.parametrize("lanes", [0, 1, 2])
def test_batched_chains_share_launches_like_plain_runs(ctd, contexts, lanes):
    # (with fewer streams than requests, chains share scratch tallies one after another)
    ps = [I.head(10_007, 6, seed=3, shape=(24, 20, 16), d=1.0), I.cbct_water(200_001, 6, seed=4, shape=(32, 30, 8), d=0.8),
          I.head(60_000, 6, seed=5, shape=(40, 38, 30), d=0.5), I.cbct_water(7_000, 6, seed=6, shape=(16, 16, 16), d=1.0),
          I.head(33_333, 6, seed=7, shape=(20, 44, 18), d=0.8)]
    c = ctd.ctd_create(device=0, batch_lanes=lanes)
    hs = [ctd.load_problem(c, p) for p in ps]
    for _ in range(2):   # recorded, then replayed
        ctd.ctd_run_batch(c, hs, [p.n_hist for p in ps], [p.seed for p in ps], 6)
        got = [ctd.ctd_get_dose_and_stddev(c, h, p.phantom.nvox) for h, p in zip(hs, ps)]
    for h, p, (dose, sd, st) in zip(hs, ps, got):
        d1, s1, t1, _ = ctd.run_problem(contexts[1], p)
        assert [st[k] for k in COUNTS] == [t1[k] for k in COUNTS]
        assert np.allclose(dose, d1, rtol=1e-12, atol=0)
    ctd.ctd_destroy(c)


@pytest.mark.parametrize("hist", [(9_001,) * 8, (900_000, 40_000, 30_011, 20_000, 9_000, 8_000, 5_003, 1_000),
                                  (2, 3, 2_000_000, 100, 5_000, 33, 2, 7)])
@pytest.mark.parametrize("threads", [0, 128])
def test_chains_on_a_third_of_the_gpu_equal_plain_runs(ctd, contexts, hist, threads):
    # eight chains: those with twice their histories still to be issued take a third of
    # the blocks (alike, falling and dominated by one), at the default and another shape
    ps = [I.head(n, 2, seed=50 + i, shape=(18 + i, 20, 14), d=1.0) for i, n in enumerate(hist)]
    c = ctd.ctd_create(device=0, threads_per_block=threads, blocks_per_sm=7 if threads else 0)
    hs = [ctd.load_problem(c, p) for p in ps]
    ctd.ctd_run_batch(c, hs, [p.n_hist for p in ps], [p.seed for p in ps], 2)
    for h, p in zip(hs, ps):
        dose, sd, st = ctd.ctd_get_dose_and_stddev(c, h, p.phantom.nvox)
        d1, s1, t1, h1 = ctd.run_problem(contexts[0], p)
        ctd.ctd_destroy_phantom(contexts[0], h1)
        assert [st[k] for k in COUNTS] == [t1[k] for k in COUNTS]
        assert np.allclose(dose, d1, rtol=1e-12, atol=0)
    ctd.ctd_destroy(c)


@pytest.mark.parametrize("n_mat,e_max", [(1, 150), (16, 150), (16, 400), (16, 780)])
def test_default_launch_shape_with_small_and_large_tables(ctd, contexts, n_mat, e_max):
    # blocks of 384 threads while three of them fit beside the attenuation tables, else
    # the 256-thread shape, up to tables that leave room for one block
    rng = np.random.default_rng(5)
    mats = [I.WATER, I.BONE, I.BRAIN, I.SOFT_TISSUE][:min(n_mat, 4)] * (4 if n_mat == 16 else 1)
    shape = (16, 18, 20)
    ph = I.Phantom(20, 18, 16, 0.5, 0.5, 0.5, rng.integers(0, n_mat, shape).astype(np.uint8),
                   rng.uniform(0.5, 2.0, shape).astype(np.float32), mats)
    p = I.Problem("tables", ph, I.arc_source(100.0, -4.0, 4.0, -3.0, 3.0, n_proj=90), I.spectrum_kramers(120, 2.5),
                  I.Physics(e_max=e_max, n_zeta=64), 40_003, 3, 9)
    explicit = ctd.ctd_create(device=0, threads_per_block=128, blocks_per_sm=1)
    (d0, _, t0, h0), (d1, _, t1, _) = (ctd.run_problem(c, p) for c in (contexts[0], explicit))
    ctd.ctd_destroy_phantom(contexts[0], h0)
    ctd.ctd_destroy(explicit)
    assert [t0[k] for k in COUNTS] == [t1[k] for k in COUNTS]
    assert np.allclose(d0, d1, rtol=1e-12, atol=0)


HI = 1 << 32   # a launch's histories share the upper word of their index


@pytest.mark.parametrize("a,b", [(HI - 3_000, HI + 2_000), (HI, HI + 1_000), (3 * HI - 1, 3 * HI + 1)])
def test_histories_across_an_upper_word(ctd, contexts, oracle, a, b):
    # records, counts and deposits of a range that a launch covers in two pieces, against
    # the binary64 oracle and against the pieces run apart
    from track_compare import compare

    p = I.head(4 * HI + 5, 7, seed=21, shape=(32, 30, 20), d=0.8)
    c = contexts[0]
    h = ctd.load_problem(c, p)
    dev = ctd.ctd_trace_range(c, h, p.n_hist, p.seed, p.n_batches, a, b)
    s = compare(dev, oracle.Setup(p, 64).track(a, b, threads=16))
    assert s["never_ended"] == 0 and s["mismatches"] <= 5e-3 * (b - a), s
    whole, parts = [], []
    for ranges, out in (([(a, b)], whole), ([(a, a + (b - a) // 3), (a + (b - a) // 3, b)], parts)):
        for k, (lo, hi) in enumerate(ranges):
            ctd.ctd_run_range(c, h, p.n_hist, p.seed, p.n_batches, lo, hi, clear=k == 0)
        _, _, st = ctd.ctd_get_dose_and_stddev(c, h, 0, want_arrays=False)
        out += [ctd.ctd_get_edep(c, h, p.phantom.nvox), [st[k] for k in COUNTS]]
    ctd.ctd_destroy_phantom(c, h)
    assert whole[1] == parts[1] and whole[1][-1] == int(dev["steps"].sum())
    assert np.allclose(whole[0], parts[0], rtol=1e-12, atol=0)


def test_groups_of_batches_of_a_large_grid(ctd, contexts):
    # 33.6 M voxels: four tallies fit side by side into the scratch memory, so five
    # batches take two launches and two folds
    p = I.cbct_water(30_001, 5, seed=13, shape=(256, 256, 512), d=0.1)
    out = []
    for c in contexts:
        dose, sd, st, h = ctd.run_problem(c, p)
        ctd.ctd_destroy_phantom(c, h)
        out.append((dose, sd, st))
    (d0, s0, t0), (d1, s1, t1) = out
    assert t0["transport_launches"] == 2 and t1["transport_launches"] == 5
    assert [t0[k] for k in COUNTS] == [t1[k] for k in COUNTS]
    assert np.allclose(d0, d1, rtol=1e-12, atol=0)
    assert np.allclose(s0 ** 2, s1 ** 2, rtol=1e-9, atol=1e-12 * float((d0 ** 2).max()))
    assert t0["avg_rsd"] == pytest.approx(t1["avg_rsd"], rel=1e-9)
    assert t0["e_deposited_kev"] == pytest.approx(t1["e_deposited_kev"], rel=1e-12)


@pytest.mark.parametrize("n_req", [1, 2, 3, 6])
def test_served_requests_sharing_the_gpu_equal_plain_runs(ctd, contexts, n_req):
    # three requests or more take a third of the blocks each; the last ones to run, and
    # fewer, all of them and, alone, smaller claims
    p = [I.head(1, seed=70 + i, shape=(18, 20, 14 + i), d=1.1) for i in range(n_req)]
    B, k = 20_011, 4
    c = ctd.ctd_create(device=0)
    hs = [ctd.load_problem(c, x) for x in p]
    ids = [ctd.ctd_submit(c, h, B, 0.0, x.seed, n_histories_max=(k + i) * B, min_batches=2)
           for i, (h, x) in enumerate(zip(hs, p))]
    for i in ids:
        assert ctd.ctd_wait(c, i, 60.0)["state"] == ctd.REQ_DONE
    for i, (h, x) in enumerate(zip(hs, p)):
        dose, sd, st = ctd.ctd_get_dose_and_stddev(c, h, x.phantom.nvox)
        d1, s1, t1, h1 = ctd.run_problem(contexts[0], I.scaled(x, n_hist=(k + i) * B, n_batches=k + i))
        ctd.ctd_destroy_phantom(contexts[0], h1)
        assert [st[q] for q in COUNTS] == [t1[q] for q in COUNTS]
        assert np.allclose(dose, d1, rtol=1e-12, atol=0)
    ctd.ctd_destroy(c)
