"""The Gabor map and the emission times on either side of the sizes up to which one thread
sums a frequency: short windows, few bins, few times, very many frequencies, and blocks of
times that reach no bin.  Against the plain sums in FP64; phases w t below 110 are rounded
once (1.5e-14 rad), sums of n <= 700 terms differ by n eps of the sum of moduli, rotations
between anchors add 64 eps: 1e-12 of that sum bounds all."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import sfhk as S

T0, DT = -35.0, 0.1


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _gabor(x, times, om, sigma):
    re, im = (torch.empty(len(times), len(om), dtype=torch.float64, device="cuda") for _ in range(2))
    S.sfhk_gabor(_dev(x), T0, DT, sigma, _dev(times), _dev(om), re, im)
    return re.cpu().numpy() + 1j * im.cpu().numpy()


def _plain(x, times, om, sigma):
    t = T0 + DT * np.arange(len(x))
    d = t - times[:, None]
    y = np.where(np.abs(d) <= 9 * sigma, np.exp(-d * d / (2 * sigma ** 2)), 0.0) * x * DT
    return y @ np.exp(1j * np.outer(t, om))


@pytest.mark.parametrize("n_times,n_omega", [(1, 1), (7, 129), (8, 20), (10, 127), (50, 1500)])
@pytest.mark.parametrize("n_bins,sigma", [(1, 5.0), (10, 5.0), (100, 5.0), (300, 5.0), (700, 0.0012), (700, 0.05), (700, 0.3),
                                          (700, 0.5), (700, 0.7), (700, 0.8), (700, 1.0)])
def test_either_side_of_the_short_windows(n_bins, sigma, n_times, n_omega):
    rng = np.random.default_rng(n_bins)
    x, om = rng.standard_normal(n_bins), rng.uniform(0.0, 3.0, n_omega)
    times = rng.uniform(T0 - 1.0, T0 + DT * n_bins + 1.0, n_times)
    times[:2] = [T0, T0 + 0.05 * n_bins][:n_times]
    got = _gabor(x, times, om, sigma)
    assert np.max(np.abs(got - _plain(x, times, om, sigma))) <= 1e-12 * np.sum(np.abs(x)) * DT


@pytest.mark.parametrize("sigma", [0.1, 5.0])
@pytest.mark.parametrize("n_omega", [20, 900])
def test_rows_without_bins_are_zero_or_nan(sigma, n_omega):
    # times of whole blocks of eight beyond the bins, some of them not numbers
    rng = np.random.default_rng(2)
    x, om = rng.standard_normal(700), rng.uniform(0.0, 3.0, n_omega)
    times = np.linspace(500.0, 600.0, 37)
    times[[0, 9, 36]] = np.nan
    times[20] = 1.0
    got = _gabor(x, times, om, sigma)
    assert np.isnan(got[[0, 9, 36]].real).all() and np.isnan(got[[0, 9, 36]].imag).all()
    rest = np.setdiff1d(np.arange(37), [0, 9, 20, 36])
    assert (got[rest] == 0.0).all()
    assert np.max(np.abs(got[20] - _plain(x, times[20:21], om, sigma)[0])) <= 1e-12 * np.sum(np.abs(x)) * DT


@pytest.mark.parametrize("n_times,n_omega", [(1, 33), (5, 1), (5, 129), (6, 129), (7, 31), (41, 20000), (42, 20000), (30, 15000),
                                             (29, 15000)])
def test_emission_times_of_either_form(n_times, n_omega):
    rng = np.random.default_rng(n_times)
    times = np.arange(n_times, dtype=float)
    p = rng.integers(0, 4, (n_times, n_omega)).astype(float)   # ties take the first time
    p[:, -1] = 0.0
    cen, peak = (torch.empty(n_omega, dtype=torch.float64, device="cuda") for _ in range(2))
    lo, hi = 0.5, n_times - 1.5
    S.sfhk_emission_time(_dev(p), _dev(np.zeros_like(p)), _dev(times), lo, hi, cen, peak)
    cen, peak = cen.cpu().numpy(), peak.cpu().numpy()
    sel = (times >= lo) & (times <= hi)
    q, t = p[sel] ** 2, times[sel]
    none = q.sum(axis=0) == 0 if q.size else np.ones(n_omega, bool)
    assert np.array_equal(np.isnan(cen), none) and np.array_equal(np.isnan(peak), none)
    if none.all():
        return
    q = q[:, ~none]
    assert np.max(np.abs(cen[~none] - (t @ q) / q.sum(axis=0))) <= 1e-12 * n_times
    j = np.argmax(q, axis=0)
    ref = t[j].copy()
    for m in np.nonzero((j > 0) & (j < len(t) - 1))[0]:
        a, b, c = q[j[m] - 1, m], q[j[m], m], q[j[m] + 1, m]
        if a > 0 and c > 0 and np.log(a) - 2 * np.log(b) + np.log(c) < 0:
            ref[m] += 0.5 * (np.log(a) - np.log(c)) / (np.log(a) - 2 * np.log(b) + np.log(c))
    assert np.max(np.abs(peak[~none] - ref)) <= 1e-12 * n_times
