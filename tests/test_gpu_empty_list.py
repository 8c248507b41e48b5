"""A mixed call in which nothing escalates: its redo launches find an empty list and return
at once.  Bins are those of the one-thread redo's call, and the time is about the same
(microseconds of launches; blocks that look through every SM's list of groups take
three times as long)."""
import pytest
import torch

from paper_2601_17164_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import pipeline as PL
    from paper_2601_17164_gb300 import sfhk as S


@pytest.mark.parametrize("target", [W.HYDROGEN, W.ARGON], ids=["H", "Ar"])
def test_an_empty_list_costs_a_launch(target):
    # births at the last grid points: next to no steps, no escalation
    w = W.Workload("t", target, W.Pulse(1.2e14, 800.0, 1.0, 0.4), dt=0.02, n=64, sigma=0.2, seed=8)
    field, tg = PL.make_handles(w)
    b = PL.sample(w, field, tg)
    b.n0.fill_(field.info["n_steps"] - 10)
    out, best = [], []
    for ep in (0, 2):
        dl = torch.zeros(field.info["n_bins"], dtype=torch.float64, device="cuda")
        dv, st = torch.zeros_like(dl), S.new_stats()
        pp = S.prop_params(S.MIXED, w.gamma, w.d_t, esc_precision=ep)
        S.sfhk_dipole(field, tg, b, len(b), pp, dl, dv, st)
        out.append((dl.clone(), dv.clone(), S.stats_dict(st)))
        t = 1e30
        for _ in range(20):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            S.sfhk_dipole(field, tg, b, len(b), pp, dl, dv, st)
            e1.record()
            torch.cuda.synchronize()
            t = min(t, e0.elapsed_time(e1))
        best.append(t)
    assert out[0][2] == out[1][2] and out[0][2]["escalated"] == 0
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert best[0] < 2.0 * best[1], best
