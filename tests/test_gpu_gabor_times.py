"""The Gabor map for any contents of the array of times and wide windows, against the plain
sum in FP64: a time that is not a number has a row of NaN and leaves its seven neighbours
in the block as they are; times far outside the bins with windows that reach them or do
not.

Weights are exponentials of sums of at most four terms of modulus 81 or less (1e-13
relative), phases w t below 110 (1.5e-14 rad), sums of n terms differ by n eps of the sum
of moduli: 1e-12 of that sum bounds all three.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import sfhk as S

N, T0, DT = 700, -35.0, 0.1


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _gabor(x, times, om, sigma, n=N):
    re, im = (torch.empty(len(times), len(om), dtype=torch.float64, device="cuda") for _ in range(2))
    S.sfhk_gabor(_dev(x[:n]), T0, DT, sigma, _dev(times), _dev(om), re, im)
    return re.cpu().numpy(), im.cpu().numpy()


def _data():
    rng = np.random.default_rng(1)
    return rng.standard_normal(N), rng.uniform(0.0, 3.0, 65)


@pytest.mark.parametrize("bad", [[3], [0], [7, 8], [0, 1, 2, 3, 4, 5, 6, 7]])
def test_a_time_that_is_not_a_number_has_a_row_of_nan(bad):
    x, om = _data()
    times = np.linspace(-10.0, 10.0, 19)
    ref = _gabor(x, times, om, 0.9)
    times[bad] = np.nan
    for a, b in zip(_gabor(x, times, om, 0.9), ref):
        good = np.setdiff1d(np.arange(19), bad)
        assert np.isnan(a[bad]).all()
        assert np.array_equal(a[good], b[good])


@pytest.mark.parametrize("sigma", [0.9, 60.0, 1e3, 1e6, 1e30])
def test_times_far_from_the_bins(sigma):
    x, om = _data()
    times = np.array([-np.inf, -1e30, -1e6, -3e3, -300.0, -36.0, 0.02, 36.0, 300.0, 3e3, 1e6, 1e30, np.inf])
    re, im = _gabor(x, times, om, sigma)
    t = T0 + DT * np.arange(N)
    with np.errstate(all="ignore"):
        d = t - times[:, None]
        y = np.where(np.abs(d) <= 9 * sigma, np.exp(-d * d / (2 * sigma ** 2)), 0.0) * x * DT
    ref = y @ np.exp(1j * np.outer(t, om))
    assert np.max(np.abs(re + 1j * im - ref)) <= 1e-12 * np.sum(np.abs(x)) * DT


def test_no_bins_is_zero_for_every_time():
    x, om = _data()
    for a in _gabor(x, np.array([0.0, np.nan, np.inf]), om, 0.9, n=0):
        assert (a == 0.0).all()
