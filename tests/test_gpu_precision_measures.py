"""The precision measures (mean s/D over D > 0.1 D_max, s/D_max over D > 0.2 D_max,
inside rho >= 0.1) of device arrays against numpy in binary64, at the edges of a
thread's four voxels, a block and the resident grid, on addresses that are only
8-byte aligned, and on values the shared-reciprocal sums must not mistake: NaN,
infinite and negative doses, doses at both ends of the binary64 range, empty masks.
A sum's terms are non-negative and each passes fewer than 100 rounded operations,
so the measures are within 100 * 2^-53 = 1.1e-14; the bound is 2e-14 with the
reference's own rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [1, 255, 256, 1023, 1024, 1025, 152 * 8 * 1024 - 1, 152 * 8 * 1024 + 1, 5_000_011]


@pytest.fixture(scope="module")
def ctd():
    from paper_1109_3266_gb300 import build, ctd as binding
    build.build()
    return binding


def reference(dose, sd, rho):
    with np.errstate(all="ignore"):
        ok = (rho >= np.float32(0.1)) & (dose > 0.0)
        dmax = dose[ok].max() if ok.any() else 0.0
        m1, m2 = ok & (dose > 0.1 * dmax), ok & (dose > 0.2 * dmax)
        avg = float((sd[m1] / dose[m1]).sum() / m1.sum()) if m1.any() else 0.0
        bar = float(sd[m2].sum() / (m2.sum() * dmax)) if m2.any() else 0.0
    return np.array([avg, bar, dmax])


def device(ctd, dose, sd, rho, offset=0):
    import torch

    def put(a):
        t = torch.zeros(a.size + offset, dtype=torch.from_numpy(a[:1]).dtype, device="cuda")
        t[offset:] = torch.from_numpy(a).cuda()
        return t

    d, s, r = put(dose), put(sd), put(rho)
    out = torch.full((3,), float("nan"), dtype=torch.float64, device="cuda")
    for _ in range(2):   # nothing is carried over from call to call
        ctd.ctd_avg_rsd_noalloc(d.data_ptr() + 8 * offset, s.data_ptr() + 8 * offset, r.data_ptr() + 4 * offset, dose.size,
                                out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def arrays(n, seed=0, scale=1e-15):
    rng = np.random.default_rng(seed)
    rho = rng.choice(np.array([0.0012, 0.0999, 0.1, 1.0], dtype=np.float32), n)
    dose = scale * rng.uniform(0.0, 1.0, n)
    return dose, dose * rng.uniform(0.001, 0.5, n), rho


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n", SIZES)
def test_sizes_and_addresses(ctd, n, offset):
    a = arrays(n, seed=n)
    np.testing.assert_allclose(device(ctd, *a, offset=offset), reference(*a), rtol=2e-14, atol=0)


@pytest.mark.parametrize("scale", [1e-320, 1e-305, 1e-290, 1.0, 1e290, 1e302])
def test_scales(ctd, scale):
    a = arrays(70_003, scale=scale)
    # (subnormal doses have few digits, the same ones on both sides)
    np.testing.assert_allclose(device(ctd, *a), reference(*a), rtol=2e-14, atol=0)


def test_special_values(ctd):
    dose, sd, rho = arrays(50_001, seed=3)
    dose[::7] = np.nan
    dose[1::7] = -dose[1::7]
    dose[2::11] = -np.inf
    rho[5::13] = np.nan
    a = (dose, sd, rho)
    np.testing.assert_allclose(device(ctd, *a), reference(*a), rtol=2e-14, atol=0)
    # an infinite dose leaves nothing above a tenth of the maximum
    dose[4] = np.inf
    rho[4] = 1.0
    assert device(ctd, *a).tolist() == [0.0, 0.0, np.inf]
    # a NaN error inside the mask shows
    dose, sd, rho = arrays(5_000, seed=4)
    k = int(np.argmax(np.where(rho >= np.float32(0.1), dose, 0.0)))
    sd[k] = np.nan
    r = device(ctd, dose, sd, rho)
    assert np.isnan(r[0]) and np.isnan(r[1]) and r[2] == dose[k]


@pytest.mark.parametrize("case", ["no_density", "no_dose"])
def test_empty_masks(ctd, case):
    dose, sd, rho = arrays(3_001)
    if case == "no_density":
        rho[:] = 0.0
    else:
        dose[:] = 0.0
    assert device(ctd, dose, sd, rho).tolist() == [0.0, 0.0, 0.0]
