"""The spectrum and Gabor kernels at the edges of their tiles against the plain sums in
FP64 (spectrum runs of 16 bins in tiles of 160 runs, 4 to 8 blocks per 32 frequencies;
Gabor blocks of 8 times and 64 frequencies, m tiles of 256).

The phases w t are rounded once in either evaluation (|w t| < 2000: 2.3e-13 rad); sums of
n terms differ by n eps of the sum of moduli at most: 1e-12 of that sum bounds both.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import sfhk as S


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n_bins,n_omega", [(1, 1), (15, 33), (16, 32), (17, 31), (2559, 40), (2561, 700), (30000, 2500)])
@pytest.mark.parametrize("tau", [0.03, 60.0, 1e4])
def test_spectrum_edges(n_bins, n_omega, tau):
    rng = np.random.default_rng(n_bins)
    t0, dt = -0.05 * n_bins, 0.1
    x, om = rng.standard_normal(n_bins), rng.uniform(0.0, 1.2, n_omega)
    re, im = (torch.empty(n_omega, dtype=torch.float64, device="cuda") for _ in range(2))
    S.sfhk_spectrum(_dev(x), t0, dt, tau, _dev(om), re, im)
    t = t0 + dt * np.arange(n_bins)
    y = np.where(np.abs(t) <= tau, 0.5 * (1 + np.cos(np.pi * t / tau)), 0.0) * x * dt
    ref = np.array([np.sum(y * np.exp(1j * w * t)) for w in om])
    assert np.max(np.abs(re.cpu().numpy() + 1j * im.cpu().numpy() - ref)) <= 1e-12 * np.sum(np.abs(x)) * dt


def test_spectrum_carries_non_finite_bins():
    x = np.ones(100)
    x[3] = np.nan   # outside the window: 0 * NaN
    re, im = (torch.empty(5, dtype=torch.float64, device="cuda") for _ in range(2))
    S.sfhk_spectrum(_dev(x), -5.0, 0.1, 1.0, _dev(np.linspace(0.1, 1, 5)), re, im)
    assert torch.isnan(re).all() and torch.isnan(im).all()


@pytest.mark.parametrize("sigma", [0.004, 0.03, 0.9, 2.84, 2.85, 40.0])
@pytest.mark.parametrize("n_times,n_omega", [(1, 1), (7, 64), (9, 65)])
def test_gabor_edges(sigma, n_times, n_omega):
    # windows of no bin, one bin, 161, 511 and 513 bins, and longer than the bins; times
    # off the grid, outside the bins and at their ends
    n, t0, dt = 700, -35.0, 0.1
    rng = np.random.default_rng(n_times)
    x, om = rng.standard_normal(n), rng.uniform(0.0, 3.0, n_omega)
    times = np.concatenate([[t0 - 8.0, t0, t0 + dt * (n - 1), 60.0], rng.uniform(-36, 36, 9)])[:n_times]
    re, im = (torch.empty(n_times, n_omega, dtype=torch.float64, device="cuda") for _ in range(2))
    S.sfhk_gabor(_dev(x), t0, dt, sigma, _dev(times), _dev(om), re, im)
    t = t0 + dt * np.arange(n)
    d = t - times[:, None]
    y = np.where(np.abs(d) <= 9 * sigma, np.exp(-d * d / (2 * sigma ** 2)), 0.0) * x * dt
    ref = y @ np.exp(1j * np.outer(t, om))
    assert np.max(np.abs(re.cpu().numpy() + 1j * im.cpu().numpy() - ref)) <= 1e-12 * np.sum(np.abs(x)) * dt


@pytest.mark.parametrize("n_times,n_omega", [(1, 1), (2, 31), (15, 33), (17, 32), (200, 70)])
def test_emission_time_edges(n_times, n_omega):
    # ties take the first time; a frequency without signal gives NaN
    times = np.arange(n_times, dtype=float)
    rng = np.random.default_rng(n_omega)
    p = rng.integers(0, 4, (n_times, n_omega)).astype(float)
    if n_omega > 1:
        p[:, -1] = 0.0
    cen, peak = (torch.empty(n_omega, dtype=torch.float64, device="cuda") for _ in range(2))
    lo, hi = 0.5, n_times - 1.5
    S.sfhk_emission_time(_dev(p), _dev(np.zeros_like(p)), _dev(times), lo, hi, cen, peak)
    sel = (times >= lo) & (times <= hi)
    for m in range(n_omega):
        q, t = p[sel, m] ** 2, times[sel]
        if q.size == 0 or q.sum() == 0:
            assert np.isnan(cen[m].item()) and np.isnan(peak[m].item())
            continue
        assert abs(cen[m].item() - np.sum(q * t) / q.sum()) <= 1e-12 * n_times
        j = int(np.argmax(q))
        ref = t[j]
        if 0 < j < q.size - 1 and q[j - 1] > 0 and q[j + 1] > 0:
            a, b, c = np.log(q[j - 1]), np.log(q[j]), np.log(q[j + 1])
            if a - 2 * b + c < 0:
                ref = t[j] + 0.5 * (a - c) / (a - 2 * b + c)
        assert abs(peak[m].item() - ref) <= 1e-12 * n_times
