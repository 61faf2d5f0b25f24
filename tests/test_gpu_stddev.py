"""The standard error of the mean, bit by bit, from tallies of known energies folded
through the sharded run's entry points: sums in the kernels' order with every
operation rounded once (fused ones too, in exact rational arithmetic) and a square
root that is the correctly rounded one.  And tallies that are not finite: a variance that
is not a number counts as none, an infinite one gives an infinite error."""
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_1109_3266_gb300 import inputs as I

pytestmark = pytest.mark.gpu

KEV_TO_J = 1.602176634e-16


@pytest.fixture(scope="module")
def ctd():
    from paper_1109_3266_gb300 import build, ctd as binding
    build.build()
    return binding


def fold(ctd, tallies, n_hist, shape):
    """dose, standard error and totals of the batch tallies [nb][nz ny nx] (keV)."""
    import torch

    nz, ny, nx = shape
    p = I.Problem("t", I.uniform_box(nx, ny, nz, 1.0), I.static_source(50.0, 1.0, 1.0), I.spectrum_line(60.0), I.Physics(),
                  n_hist, len(tallies), 1)
    c = ctd.ctd_create(device=0)
    h = ctd.load_problem(c, p)
    ctd.ctd_shard_begin(c, h, n_hist, 1, len(tallies))
    for b, t in enumerate(tallies):
        buf = torch.from_numpy(np.ascontiguousarray(t, dtype=np.float64)).cuda()
        torch.cuda.synchronize()
        ctd.ctd_shard_fold(c, h, b, buf.data_ptr())
        ctd.ctd_shard_counts(c, h)   # waited for: the buffer goes
    counts, energies = ctd.ctd_shard_counts(c, h)
    ctd.ctd_shard_finish(c, h, counts, energies)
    dose, sd, st = ctd.ctd_get_dose_and_stddev(c, h, p.phantom.nvox)
    ctd.ctd_destroy(c)
    return dose, sd, st


def fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))   # rounded once, to nearest even


def root(x):
    """sqrt(x) correctly rounded (math.sqrt is, by IEEE 754), 0 for x <= 0."""
    return math.sqrt(x) if x > 0.0 else 0.0


@pytest.mark.parametrize("n_hist,nb", [(1000, 2), (100_003, 3), (7_000_000, 5)])
def test_bit_for_bit(ctd, n_hist, nb):
    shape = (10, 20, 30)
    nv = 10 * 20 * 30
    rng = np.random.default_rng(nb)
    # energies over many binades, close and far batches, and voxels without any
    base = np.exp(rng.uniform(-12, 20, nv))
    tallies = [base * (1.0 + rng.choice([1e-9, 1e-3, 1.0, 30.0], nv) * rng.random(nv)) for _ in range(nb)]
    for t in tallies:
        t[::17] = 0.0
        t[rng.random(nv) < 0.1] = 0.0
    dose, sd, _ = fold(ctd, tallies, n_hist, shape)
    inv_nb, inv_nn = 1.0 / nb, 1.0 / (float(nb) * (nb - 1))
    n_lo, rem = divmod(n_hist, nb)
    for v in range(nv):
        s1 = s2 = 0.0
        for b in range(nb):
            w = KEV_TO_J * 1000.0 / (1.0 * float(n_lo + (b < rem)))   # water of 1 g/cm^3, 1 cm^3
            t = float(tallies[b][v])
            s1, s2 = fma(w, t, s1), fma(w * w, t * t, s2)
        D = s1 * inv_nb
        assert dose[v] == D
        assert sd[v] == root(fma(-D, s1, s2) * inv_nn), v


def test_tallies_that_are_not_finite(ctd):
    # batches whose sum and sum of squares are infinite, or not numbers
    a = np.ones((2, 8))
    a[0, 1] = np.inf            # sum and squares infinite: no variance
    a[:, 2] = np.inf
    a[1, 3] = np.nan
    a[0, 4], a[1, 4] = 1e250, 3e250   # only the sum of squares overflows
    a[:, 5] = 0.0
    a[0, 6], a[1, 6] = 1.0, 3.0
    dose, sd, _ = fold(ctd, a, 1000, (2, 2, 2))
    assert dose[1] == np.inf and dose[2] == np.inf and np.isnan(dose[3])
    assert sd[[1, 2, 3]].tolist() == [0.0, 0.0, 0.0]
    assert sd[4] == np.inf
    assert dose[5] == 0.0 and sd[5] == 0.0
    w = KEV_TO_J * 1000.0 / 500.0
    assert sd[6] == pytest.approx(w, rel=1e-14) and dose[6] == pytest.approx(2.0 * w, rel=1e-15)
