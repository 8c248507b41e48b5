"""FP64 calls at the length from which the one-thread-per-trajectory kernel takes them
(endpoints: 13 groups of 32 per SM for Tong-Lin, 34 for the other potentials; dipoles of
the harmonic potential: 16): on either side of it the results are those of that kernel,
which a caller's own block size asks for.  Below it the same operations on other warps:
endpoints to 1e-13 of their largest entry, bins to the order of their sums (78,000 terms
differ by 9e-12 of the sum of moduli at most; 1e-10 of the largest bin leaves a decade of
cancellation); above it endpoints are equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_2601_17164_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import pipeline as PL
    from paper_2601_17164_gb300 import sfhk as S

HARMONIC = W.Target("harmonic", W.POT_HARMONIC, (0.2,), 0.5, 0, tuple(W.H_C), tuple(W.H_ALPHA))


def _sample(target, n):
    # 400 steps: the length of the call decides, not that of the pulse
    w = W.Workload("t", target, W.Pulse(1.2e14, 300.0, 1.0, 0.4), dt=0.1, n=n, sigma=0.2, seed=8)
    field, tg = PL.make_handles(w)
    return field, tg, PL.sample(w, field, tg)


@pytest.mark.parametrize("target,groups", [(W.ARGON, 13), (W.HYDROGEN, 34), (HARMONIC, 34)], ids=["Ar", "H", "harmonic"])
@pytest.mark.parametrize("over", [0, 1])
def test_endpoints_on_either_side(target, groups, over):
    n = 32 * groups * torch.cuda.get_device_properties(0).multi_processor_count + over
    field, tg, b = _sample(target, n)
    out = []
    for kw in ({}, {"block": 128}):
        st = S.new_stats()
        y, c, fl = S.sfhk_propagate(field, tg, b, n, S.prop_params(S.FP64, 0.5, 1e3, **kw), field.info["n_steps"], st)
        out.append((torch.cat([y, torch.view_as_real(c).T]), fl, S.stats_dict(st)))
    (y0, f0, s0), (y1, f1, s1) = out
    assert torch.equal(f0, f1) and s0 == s1
    assert torch.equal(torch.isnan(y0), torch.isnan(y1))
    if over:
        assert torch.equal(torch.nan_to_num(y0), torch.nan_to_num(y1))
    fin = torch.isfinite(y1).all(dim=0)
    scale = y1[:, fin].abs().amax(dim=0).clamp(min=1.0)
    assert ((y0 - y1)[:, fin].abs() / scale).max().item() <= 1e-13


@pytest.mark.parametrize("over", [0, 1])
def test_harmonic_dipole_on_either_side(over):
    n = 32 * 16 * torch.cuda.get_device_properties(0).multi_processor_count + over
    field, tg, b = _sample(HARMONIC, n)
    out = []
    for kw in ({}, {"block": 128}):
        dl = torch.zeros(field.info["n_bins"], dtype=torch.float64, device="cuda")
        dv, st = torch.zeros_like(dl), S.new_stats()
        S.sfhk_dipole(field, tg, b, n, S.prop_params(S.FP64, 0.5, 1e30, **kw), dl, dv, st)
        out.append((dl.cpu().numpy(), dv.cpu().numpy(), S.stats_dict(st)))
    assert out[0][2] == out[1][2]
    for x, y in zip(out[0][:2], out[1][:2]):
        assert np.max(np.abs(x - y)) <= 1e-10 * np.max(np.abs(y))
