"""FP64 endpoints on the eight-warp kernel against the one-thread-per-trajectory kernel:
every value is formed by the same operations, so regular trajectories agree to the last
bits (1e-13 of the largest entry allows for a fused operation in one of them carried over
some hundred steps); flags and counters are equal.  Edges: group sizes around 32, births
at and after the end point, removal at the first bins, bins at every step, births off the
axis."""
import numpy as np
import pytest
import torch

from paper_2601_17164_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import pipeline as PL
    from paper_2601_17164_gb300 import sfhk as S

HARMONIC = W.Target("harmonic", W.POT_HARMONIC, (0.2,), 0.5, 0, tuple(W.H_C), tuple(W.H_ALPHA))
ZERO = W.Target("free", W.POT_ZERO, (), 0.5, 0, tuple(W.H_C), tuple(W.H_ALPHA))


@pytest.mark.parametrize("target", [W.HYDROGEN, W.ARGON, HARMONIC, ZERO], ids=lambda t: t.name)
@pytest.mark.parametrize("n,frac,t_out,d_t", [(1, 1.0, 0.1, 1e30), (31, 0.4, 0.1, 1e30), (33, 1.0, 0.02, 1e30),
                                              (70, 0.7, 0.02, 3.0), (64, 0.0, 0.1, 1e30)])
def test_endpoints_equal_one_thread_per_trajectory(target, n, frac, t_out, d_t):
    w = W.Workload("t", target, W.Pulse(1.2e14, 600.0, 1.0, 0.4), dt=0.02, t_out=t_out, n=n, sigma=0.2, seed=8)
    field, tg = PL.make_handles(w)
    b = PL.sample(w, field, tg)
    if n == 33:
        b.q0x, b.q0y = (torch.linspace(-1, 1, n, dtype=torch.float64, device="cuda") * s for s in (1.0, 0.5))
    n_end = int(frac * field.info["n_steps"])
    out = []
    for kw in ({}, {"block": 128}):
        st = S.new_stats()
        y, c, fl = S.sfhk_propagate(field, tg, b, n, S.prop_params(S.FP64, 0.5, d_t, **kw), n_end, st)
        out.append((y.cpu().numpy(), c.cpu().numpy(), fl.cpu().numpy(), S.stats_dict(st)))
    (y0, c0, f0, s0), (y1, c1, f1, s1) = out
    assert np.array_equal(f0, f1) and s0 == s1
    if d_t == 3.0 and target is not HARMONIC:
        assert s0["removed"] > 0
    # a birth without a saddle starts at the origin, where the Tong-Lin force is not a number
    fin = np.isfinite(y1).all(axis=0)
    assert np.array_equal(np.isnan(y0), np.isnan(y1)) and np.array_equal(np.isnan(c0), np.isnan(c1))
    if fin.any():
        y0, y1, c0, c1 = y0[:, fin], y1[:, fin], c0[fin], c1[fin]
        scale = np.maximum(1.0, np.max(np.abs(y1), axis=0))
        assert np.max(np.abs(y0 - y1) / scale) <= 1e-13
        assert np.max(np.abs(c0 - c1) / np.maximum(1.0, np.abs(c1))) <= 1e-12
