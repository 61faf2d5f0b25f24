"""The precision measures with doses near the ends of binary64's range, where products of
several doses and errors leave it: errors of 1e-9 to 1e-2 of the dose and of up to 1e6
doses, in many voxels and in so few that one's rounding shows.  Every term is within 3
rounded operations of s/D and the sums within 100, so 2e-14 holds as for ordinary doses."""
import numpy as np
import pytest

from test_gpu_precision_measures import ctd, device, reference  # noqa: F401  (ctd: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 20_011])
@pytest.mark.parametrize("rel", [1e-9, 1e-6, 1e-2, 1e6])
@pytest.mark.parametrize("exponent", [-960, -980, -990, -999, -1000, -1001, -501, -500, -499, 499, 500, 501, 980, 1000])
def test_scales_of_doses_and_errors(ctd, exponent, rel, n):  # noqa: F811
    rng = np.random.default_rng(exponent + 2000)
    rho = rng.choice(np.array([0.05, 1.0], dtype=np.float32), n)
    rho[:4] = 1.0
    # the largest dose lies in [2^exponent, 2^(exponent + 1))
    dose = np.ldexp(rng.uniform(0.05, 1.9, n), exponent)
    a = (dose, dose * rel * rng.uniform(0.5, 1.0, n), rho)
    np.testing.assert_allclose(device(ctd, *a), reference(*a), rtol=2e-14, atol=0)
