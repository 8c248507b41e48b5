"""The autotuner on FP64 dipoles: the planar call into atomic bins runs by default on
kernels that take no launch shape, so where that is the faster call the choice is
block = chunk_steps = 0, with that call's time; asking for a choice never makes the call
slower than not asking.  Calls that use a shape get one."""
import pytest
import torch

from paper_2601_17164_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import pipeline as PL
    from paper_2601_17164_gb300 import sfhk as S


def _time(fn):
    fn()
    best = 1e30
    for _ in range(3):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("kw,shape", [({}, False), (dict(geometry=1), True), (dict(deterministic=1), True),
                                      (dict(d_t=1e300), True)])
def test_autotune_returns_the_faster_call(kw, shape):
    # (the free potential: the shapes kept for the others stay as other tests expect them)
    free = W.Target("free", W.POT_ZERO, (), 0.5, 0, tuple(W.H_C), tuple(W.H_ALPHA))
    w = W.Workload("t", free, W.Pulse(1.2e14, 400.0, 1.0, 0.4), dt=0.02, n=3000, sigma=0.2, seed=8)
    f, t = PL.make_handles(w)
    b = PL.sample(w, f, t)
    kw = dict(dict(gamma=0.5, d_t=1e30), **kw)
    block, chunk, ms = S.sfhk_autotune(f, t, b, len(b), S.prop_params(S.FP64, **kw))
    assert ms > 0 and chunk % f.info["n_out"] == 0
    assert (block in (64, 128) and chunk > 0) if shape else (block, chunk) == (0, 0)
    dl = torch.zeros(f.info["n_bins"], dtype=torch.float64, device="cuda")
    dv = torch.zeros_like(dl)
    chosen = S.prop_params(S.FP64, **kw, block=block, chunk_steps=chunk)
    default = S.prop_params(S.FP64, **kw)
    t_c, t_d = (_time(lambda: S.sfhk_dipole(f, t, b, len(b), p, dl, dv)) for p in (chosen, default))
    assert t_c <= 2.0 * t_d, (t_c, t_d)   # (the one-thread kernel takes 2.7 times the default call's time)
