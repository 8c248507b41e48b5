"""The four-lane FP64 kernel (lists up to 8 trajectories a block) against the
one-thread-per-trajectory kernel: FP64 dipole calls and escalation lists at the edges of
its blocks and of its range, for every potential.

Both kernels form every value of a trajectory by the same operations in FP64, so bins
differ by the order of the sums over trajectories (and, in FP64 bins, over GTO terms):
n terms summed in another order differ by at most about n eps of the sum of moduli;
1e-12 of the largest bin allows for cancellation of three digits at n ~ 10^3.
Counters are equal.
"""
import numpy as np
import pytest
import torch

from paper_2601_17164_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import pipeline as PL
    from paper_2601_17164_gb300 import sfhk as S

HARMONIC = W.Target("harmonic", W.POT_HARMONIC, (0.2,), 0.5, 0, tuple(W.H_C), tuple(W.H_ALPHA))
ZERO = W.Target("free", W.POT_ZERO, (), 0.5, 1, tuple(W.AR_C), tuple(W.AR_ALPHA))


def _dipole(w, n, pp):
    field, target = PL.make_handles(w)
    births = PL.sample(w, field, target)
    dl = torch.zeros(field.info["n_bins"], dtype=torch.float64, device="cuda")
    dv, st = torch.zeros_like(dl), S.new_stats()
    S.sfhk_dipole(field, target, births, n, pp, dl, dv, st)
    return dl.cpu().numpy(), dv.cpu().numpy(), S.stats_dict(st)


def _same(a, b):
    for x, y in zip(a[:2], b[:2]):
        assert np.max(np.abs(x - y)) <= 1e-12 * np.max(np.abs(y)), np.max(np.abs(x - y)) / np.max(np.abs(y))
    assert a[2] == b[2]


@pytest.mark.parametrize("target", [W.HYDROGEN, W.ARGON, HARMONIC, ZERO], ids=lambda t: t.name)
@pytest.mark.parametrize("n", [1, 7, 8, 9, 61])
def test_fp64_dipole_equals_one_thread_per_trajectory(target, n):
    w = W.Workload("t", target, W.Pulse(1.2e14, 800.0, 1.0, 0.4), dt=0.02, n=96, sigma=0.2, seed=5)
    kw = dict(gamma=0.5, d_t=1e30)
    _same(_dipole(w, n, S.prop_params(S.FP64, **kw)), _dipole(w, n, S.prop_params(S.FP64, block=128, **kw)))


@pytest.mark.parametrize("n", [2431, 2432, 2433])
def test_fp64_dipole_at_the_limit_of_short_lists(n):
    # 2 blocks of 8 per SM on 152 SMs: 2432 births take the four-lane kernel, 2433 do not;
    # with removal and partial waves
    w = W.Workload("t", W.HYDROGEN, W.Pulse(1.2e14, 600.0, 1.0, 0.4), dt=0.02, n=2500, sigma=0.2, seed=6)
    kw = dict(gamma=0.5, d_t=30.0, pw_mask=3)
    a, b = _dipole(w, n, S.prop_params(S.FP64, **kw)), _dipole(w, n, S.prop_params(S.FP64, block=128, **kw))
    assert a[2]["removed"] > 0
    _same(a, b)


@pytest.mark.parametrize("target,n", [(W.HYDROGEN, 700), (W.ARGON, 300)], ids=["H", "Ar"])
def test_short_escalation_lists_equal_the_one_thread_redo(target, n):
    w = W.Workload("t", target, W.Pulse(1.5e14, 800.0, 3.0, 0.3), dt=0.02, n=n, sigma=0.2, seed=7)
    kw = dict(gamma=0.5, d_t=1e30, esc_ratio=2.0, esc_floor=0.0)
    a = _dipole(w, n, S.prop_params(S.MIXED, **kw))
    b = _dipole(w, n, S.prop_params(S.MIXED, esc_precision=2, **kw))
    assert 8 < a[2]["escalated"] < 2432
    _same(a, b)
