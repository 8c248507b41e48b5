"""The spectrum on either side of the number of bins up to which one thread sums a frequency
(80 to 900 by the number of frequencies): against the plain sum in FP64.  Phases w t below
200 are rounded once (2.3e-14 rad), sums of n <= 1000 terms differ by n eps of the sum of
moduli, rotations between anchors add 64 eps: 1e-12 of that sum bounds all."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import sfhk as S


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n_bins,n_omega", [(0, 3), (1, 129), (64, 20), (65, 127), (80, 1920), (81, 1920), (208, 5000),
                                            (209, 5000), (450, 20000), (451, 20000), (1000, 240000), (1001, 240000)])
@pytest.mark.parametrize("tau", [0.03, 2.0, 1e4])
def test_either_side_of_the_short_sums(n_bins, n_omega, tau):
    rng = np.random.default_rng(n_bins)
    t0, dt = -0.05 * n_bins, 0.1
    x, om = rng.standard_normal(n_bins), rng.uniform(0.0, 1.2, n_omega)
    re, im = (torch.empty(n_omega, dtype=torch.float64, device="cuda") for _ in range(2))
    S.sfhk_spectrum(_dev(x), t0, dt, tau, _dev(om), re, im)
    t = t0 + dt * np.arange(n_bins)
    y = np.where(np.abs(t) <= tau, 0.5 * (1 + np.cos(np.pi * t / tau)), 0.0) * x * dt
    pick = rng.integers(0, n_omega, 300)
    ref = np.exp(1j * np.outer(om[pick], t)) @ y
    got = re.cpu().numpy() + 1j * im.cpu().numpy()
    assert np.isfinite(got).all()
    assert np.max(np.abs(got[pick] - ref)) <= 1e-12 * np.sum(np.abs(x)) * dt


def test_short_sums_carry_non_finite_bins():
    x = np.ones(40)
    x[3] = np.inf   # outside the window: 0 * inf
    re, im = (torch.empty(5, dtype=torch.float64, device="cuda") for _ in range(2))
    S.sfhk_spectrum(_dev(x), -2.0, 0.1, 1.0, _dev(np.linspace(0.1, 1, 5)), re, im)
    assert torch.isnan(re).all() and torch.isnan(im).all()
