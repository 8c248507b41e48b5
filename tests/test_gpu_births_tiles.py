"""Births at the edges of the kernel's tiles (128 births, 512 in calls of 155648 births or
more) and of its queue: a sample's parts, produced by calls of other sizes, are the same
births bit for bit, for every amplitude and both samplers.  (Element by element against
the oracle: test_gpu_parity.py, test_gpu_variants.py.)"""
import pytest
import torch

from paper_2601_17164_gb300 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import pipeline as PL
    from paper_2601_17164_gb300 import sfhk as S

KEYS = ("n0", "t0", "p0x", "p0y", "p0z", "q0z", "amp_re", "amp_im")


@pytest.mark.parametrize("amp", [0, 1, 2])
@pytest.mark.parametrize("n", [155_647, 155_648, 156_161])
def test_tiles_give_the_same_births(amp, n):
    w = W.Workload("t", W.HYDROGEN if amp else W.ARGON, W.Pulse(1.2e14, 900.0, 3.0, 0.7), dt=0.02, n=n, sigma=0.2, seed=3)
    field, target = PL.make_handles(w, amp)
    whole = PL.sample(w, field, target)
    for first, count in ((0, 1), (127, 130), (511, 514), (n // 2, 1000), (n - 513, 513)):
        part = S.Births.empty(count)
        S.sfhk_sample_births(field, target, w.birth_mode, n, part, sigma_k=w.sigma, seed=w.seed, first=first, count=count)
        for k in KEYS:
            assert torch.equal(getattr(part, k), getattr(whole, k)[first:first + count]), (k, first)
