"""Calls in which removal ends every trajectory of a group before the pulse does: the
warp-specialised FP64 kernels end the group there, with the results, flags and counters of
the one-thread-per-trajectory kernel (the same operations: bins to the order of their sums,
1e-12 of the largest; endpoints of removed trajectories to 1e-13 of their largest entry),
and no longer than a few of its times."""
import numpy as np
import pytest
import torch

from paper_2601_17164_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import pipeline as PL
    from paper_2601_17164_gb300 import sfhk as S

KEYS = ("n0", "t0", "p0x", "p0y", "p0z", "q0z", "amp_re", "amp_im")


def _sample(target, n, t_out=0.1, shuffle=False, lam=600.0):
    w = W.Workload("t", target, W.Pulse(1.2e14, lam, 1.0, 0.4), dt=0.02, t_out=t_out, n=n, sigma=0.2, seed=8)
    field, tg = PL.make_handles(w)
    b = PL.sample(w, field, tg)
    if shuffle:   # groups whose early births are removed before their late ones start
        p = torch.randperm(n, generator=torch.Generator().manual_seed(1)).cuda()
        b = S.Births(*(getattr(b, k)[p].contiguous() for k in KEYS))
    return field, tg, b


def _dipole(field, tg, b, n, pp):
    dl = torch.zeros(field.info["n_bins"], dtype=torch.float64, device="cuda")
    dv, st = torch.zeros_like(dl), S.new_stats()
    S.sfhk_dipole(field, tg, b, n, pp, dl, dv, st)
    return dl.cpu().numpy(), dv.cpu().numpy(), S.stats_dict(st)


def _same(a, b):
    assert a[2] == b[2], (a[2], b[2])
    for x, y in zip(a[:2], b[:2]):
        assert np.max(np.abs(x - y)) <= 1e-12 * np.max(np.abs(y))


@pytest.mark.parametrize("target", [W.HYDROGEN, W.ARGON], ids=["H", "Ar"])
@pytest.mark.parametrize("n,t_out,shuffle", [(5, 0.1, False), (61, 0.02, False), (300, 0.1, True), ("wide", 0.1, False),
                                             ("wide", 0.02, True)])
@pytest.mark.parametrize("d_t", [1.5, 10.0])
def test_dipole_with_every_trajectory_removed(target, n, t_out, shuffle, d_t):
    if n == "wide":   # longer than a short list (8 times 2 or 5 groups per SM)
        n = 8 * 5 * torch.cuda.get_device_properties(0).multi_processor_count + 45
    field, tg, b = _sample(target, n, t_out, shuffle)
    kw = dict(gamma=0.5, d_t=d_t)
    out = [_dipole(field, tg, b, n, S.prop_params(S.FP64, **kw, **k)) for k in ({}, {"block": 128})]
    assert out[0][2]["removed"] > 0.5 * (n - out[0][2]["skipped"])
    _same(*out)


@pytest.mark.parametrize("target", [W.HYDROGEN, W.ARGON], ids=["H", "Ar"])
def test_redo_with_removal(target):
    field, tg, b = _sample(target, 3000, lam=800.0)
    kw = dict(gamma=0.5, d_t=200.0, esc_ratio=1.2, esc_floor=0.0, esc_big=0.0)
    out = [_dipole(field, tg, b, 3000, S.prop_params(S.MIXED, **kw, esc_precision=e)) for e in (0, 2)]
    assert out[0][2]["escalated"] > 0 and out[0][2]["removed"] > 0
    _same(*out)


@pytest.mark.parametrize("target", [W.HYDROGEN, W.ARGON], ids=["H", "Ar"])
@pytest.mark.parametrize("n,t_out,shuffle", [(5, 0.1, False), (64, 0.02, False), (1000, 0.1, True)])
def test_endpoints_with_every_trajectory_removed(target, n, t_out, shuffle):
    field, tg, b = _sample(target, n, t_out, shuffle)
    n_end = int(0.8 * field.info["n_steps"])
    b.n0[2::7] = n_end + 1   # births that never start, in groups that end early
    b.n0[3::7] = -1
    out = []
    for kw in ({}, {"block": 128}):
        st = S.new_stats()
        y, c, fl = S.sfhk_propagate(field, tg, b, n, S.prop_params(S.FP64, 0.5, 1.5, **kw), n_end, st)
        out.append((y.cpu().numpy(), c.cpu().numpy(), fl.cpu().numpy(), S.stats_dict(st)))
    (y0, c0, f0, s0), (y1, c1, f1, s1) = out
    assert np.array_equal(f0, f1) and s0 == s1 and s0["removed"] > 0 and s0["skipped"] > 0
    assert np.array_equal(np.isnan(y0), np.isnan(y1)) and np.array_equal(np.isnan(c0), np.isnan(c1))
    fin = np.isfinite(y1).all(axis=0)
    scale = np.maximum(1.0, np.max(np.abs(y1[:, fin]), axis=0))
    assert np.max(np.abs(y0[:, fin] - y1[:, fin]) / scale) <= 1e-13
    assert np.max(np.abs(c0[fin] - c1[fin]) / np.maximum(1.0, np.abs(c1[fin]))) <= 1e-12


def _time(fn):
    fn()
    best = 1e30
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("call", ["dipole", "endpoints"])
def test_removal_ends_a_call_early(call):
    n = 20_000
    field, tg, b = _sample(W.HYDROGEN, n, lam=800.0)
    dl = torch.zeros(field.info["n_bins"], dtype=torch.float64, device="cuda")
    dv = torch.zeros_like(dl)
    t = []
    for kw in ({}, {"block": 128}):
        pp = S.prop_params(S.FP64, 0.5, 1.5, **kw)
        if call == "dipole":
            t.append(_time(lambda: S.sfhk_dipole(field, tg, b, n, pp, dl, dv)))
        else:
            t.append(_time(lambda: S.sfhk_propagate(field, tg, b, n, pp, field.info["n_steps"])))
    assert t[0] < 3.0 * t[1], t
