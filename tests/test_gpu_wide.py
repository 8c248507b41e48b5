"""The four-warp FP64 kernel with 32 trajectories a block, against the one-thread-per-
trajectory kernel: FP64 dipoles and escalation lists longer than those that the four-lane
kernel takes (2 groups of 8 per SM, 5 for Tong-Lin; counted from the device's SMs), for
every potential, bins at every fifth and at every step, removal and partial waves.

Every value of a trajectory is formed by the same operations, so counters are equal and
bins differ by the order of their sums: n <= 10^4 terms differ by n eps = 1.1e-12 of the
sum of moduli, 1e-11 of the largest bin leaves a decade of cancellation."""
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
TARGETS = [W.HYDROGEN, W.ARGON, HARMONIC, ZERO]


def _limit(target):
    return 8 * torch.cuda.get_device_properties(0).multi_processor_count * (5 if target is W.ARGON else 2)


def _dipole(w, n, pp):
    field, target = PL.make_handles(w)
    births = PL.sample(w, field, target)
    dl = torch.zeros(field.info["n_bins"], dtype=torch.float64, device="cuda")
    dv, st = torch.zeros_like(dl), S.new_stats()
    S.sfhk_dipole(field, target, births, n, pp, dl, dv, st)
    return dl.cpu().numpy(), dv.cpu().numpy(), S.stats_dict(st)


def _same(a, b):
    assert a[2] == b[2], (a[2], b[2])
    for x, y in zip(a[:2], b[:2]):
        assert np.max(np.abs(x - y)) <= 1e-11 * np.max(np.abs(y)), np.max(np.abs(x - y)) / np.max(np.abs(y))


@pytest.mark.parametrize("target", TARGETS, ids=lambda t: t.name)
@pytest.mark.parametrize("over,t_out,kw", [(0, 0.1, {}), (1, 0.1, {}), (33, 0.02, {}), (1, 0.1, dict(d_t=30.0)),
                                           (17, 0.02, dict(d_t=30.0, pw_mask=6)), (1, 0.1, dict(pw_mask=1, pw_radius=2.0))])
def test_fp64_dipole_around_the_limit_of_short_lists(target, over, t_out, kw):
    n = _limit(target) + over   # 0: the four-lane kernel's longest call
    w = W.Workload("t", target, W.Pulse(1.2e14, 400.0, 1.0, 0.4), dt=0.02, t_out=t_out, n=n, sigma=0.2, seed=6)
    kw = dict(dict(gamma=0.5, d_t=1e30), **kw)
    _same(_dipole(w, n, S.prop_params(S.FP64, **kw)), _dipole(w, n, S.prop_params(S.FP64, block=128, **kw)))


@pytest.mark.parametrize("target", TARGETS, ids=lambda t: t.name)
@pytest.mark.parametrize("t_out,kw", [(0.1, {}), (0.02, {}), (0.1, dict(d_t=1e3)), (0.1, dict(pw_mask=2)),
                                      (0.02, dict(d_t=1e3, pw_mask=6))])
def test_long_escalation_lists(target, t_out, kw):
    # a growth ratio below every trajectory's: nearly all births are redone
    n = int(1.6 * _limit(target)) + 300
    w = W.Workload("t", target, W.Pulse(1.5e14, 400.0, 1.0, 0.3), dt=0.02, t_out=t_out, n=n, sigma=0.2, seed=7)
    kw = dict(dict(gamma=0.5, d_t=1e30, esc_ratio=1e-6, esc_floor=0.0, esc_big=0.0), **kw)
    a = _dipole(w, n, S.prop_params(S.MIXED, **kw))
    b = _dipole(w, n, S.prop_params(S.MIXED, esc_precision=2, **kw))
    assert a[2]["escalated"] > _limit(target)
    _same(a, b)
