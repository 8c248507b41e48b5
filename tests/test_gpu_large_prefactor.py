"""FP64 dipoles with |det Z| near and past the root of FP64's range (1.3e154), where its
square and the products that follow the branch overflow: a d_t above 1e154 is accepted and
keeps such trajectories, and a large gamma makes det Z ~ gamma^3 as large as wished.  Calls
in the sizes of the warp-specialised kernels (four-lane and 32-wide), which take d_t up to
1e150, against the one-thread-per-trajectory kernel: every value is formed by the same
operations, so bins differ by the order of the sums over trajectories only (1e-12 of the
largest bin, as in test_gpu_quad.py) and counters are equal."""
import numpy as np
import pytest
import torch

from paper_2601_17164_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import pipeline as PL
    from paper_2601_17164_gb300 import sfhk as S


@pytest.mark.parametrize("wide", [False, True], ids=["four-lane", "32-wide"])
@pytest.mark.parametrize("d_t", [1e150, 1e300])
@pytest.mark.parametrize("gamma", [1e30, 1e49, 3e49, 1e50, 1e51, 1e53, 1e60, 1e90, 1e100])
def test_large_prefactors_equal_one_thread_per_trajectory(gamma, d_t, wide):
    n = 16 * torch.cuda.get_device_properties(0).multi_processor_count + 1 if wide else 61
    w = W.Workload("t", W.HYDROGEN, W.Pulse(1.2e14, 300.0, 1.0, 0.4), dt=0.02, n=n, sigma=0.2, seed=5)
    field, target = PL.make_handles(w)
    births = PL.sample(w, field, target)
    out = []
    for kw in ({}, {"block": 128}):
        dl = torch.zeros(field.info["n_bins"], dtype=torch.float64, device="cuda")
        dv, st = torch.zeros_like(dl), S.new_stats()
        S.sfhk_dipole(field, target, births, n, S.prop_params(S.FP64, gamma, d_t, **kw), dl, dv, st)
        out.append((dl.cpu().numpy(), dv.cpu().numpy(), S.stats_dict(st)))
    (l0, v0, s0), (l1, v1, s1) = out
    assert s0 == s1, (s0, s1)
    for a, b in ((l0, l1), (v0, v1)):
        assert np.isfinite(b).all() and (np.max(np.abs(b)) > 0.0 or d_t < 1e300)
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b)), (np.max(np.abs(a - b)), np.max(np.abs(b)))
