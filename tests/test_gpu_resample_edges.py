"""Resampling at the edges of its 1024-entry blocks and of its shortcuts, bit for bit
against the oracle: pools whose amplitudes are near underflow or span 300 decades (the
threshold below which no root is taken), equal weights, n far above and below m."""
import numpy as np
import pytest
import torch

from oracle import resample as RS

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_17164_gb300 import sfhk as S

KEYS = (("n0", "n0"), ("t0", "t0"), ("px", "p0x"), ("py", "p0y"), ("pz", "p0z"), ("qz", "q0z"),
        ("amp_re", "amp_re"), ("amp_im", "amp_im"))


@pytest.mark.parametrize("m", [1, 2, 1023, 1024, 1025, 2049])
@pytest.mark.parametrize("n", [1, 700, 5000])
@pytest.mark.parametrize("kind", ["equal", "tiny", "wide", "one"])
def test_resample_edges_bit_exact(m, n, kind):
    rng = np.random.default_rng(m + n)
    a = rng.standard_normal(m) + 1j * rng.standard_normal(m)
    if kind == "equal":
        a = np.full(m, 0.3 - 0.4j)
    elif kind == "tiny":
        a = a * 1e-158
    elif kind == "wide":
        a = a * 10.0 ** rng.uniform(-170, 130, m)
    elif kind == "one":
        a = np.where(np.arange(m) == m - 1, a, 0.0)
    pool = {k: rng.standard_normal(m) for k, _ in KEYS}
    pool.update(n0=np.sort(rng.integers(1, 1000, m)).astype(np.int32), amp_re=a.real.copy(), amp_im=a.imag.copy())
    out = S.Births.empty(n)
    nd = torch.zeros(1, dtype=torch.int64, device="cuda")
    S.sfhk_resample_births(S.Births(*(torch.tensor(pool[k], device="cuda") for k, _ in KEYS)), m, n, 11, out, nd)
    ref, r = RS.resample(pool, n, 11)
    assert int(nd.item()) == r
    for k, g in KEYS:
        assert np.array_equal(getattr(out, g).cpu().numpy().view(np.uint8), ref[k].view(np.uint8)), k
