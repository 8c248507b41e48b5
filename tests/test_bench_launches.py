"""The exact number of kernel launches of a benchmark step (host-side logic of bench.py):
every schedule and escalation precision, with parts of more and of no more births than a
short list holds."""
import bench
from paper_2601_17164_gb300 import workloads as W


def _count(n, **kw):
    return bench.launches_per_step(n, 88256, 1000, 1, True, short=2432, **kw)


def test_short_list_by_potential_and_device():
    assert bench.short_list(W.POT_SOFTCORE, 152) == 2432 and bench.short_list(W.POT_TONGLIN, 152) == 6080
    assert bench.short_list(W.POT_HARMONIC, 148) == 2368 and bench.short_list(W.POT_ZERO, 148) == 2368


def test_sequential_step():
    # births, amplitude maximum, float pass, count, scatter, then the redo, two spectra
    assert _count(1_000_000, overlap=2) == 2 + 3 + 3 + 2      # plan, short and long lists
    assert _count(2433, overlap=2) == 2 + 3 + 3 + 2
    assert _count(2432, overlap=2) == 2 + 3 + 2 + 2           # no list can be long
    for ep in (1, 2):
        assert _count(1_000_000, overlap=2, esc_precision=ep) == 2 + 3 + 1 + 2
    # no amplitude floor: no maximum
    assert bench.launches_per_step(10_000, 88256, 1000, 1, False, overlap=2, short=2432) == 1 + 3 + 3 + 2


def test_birth_chunks():
    assert _count(1_000_000, overlap=0) == 2 + 8 * 6 + 2
    assert _count(1_000_000, overlap=0, esc_precision=1) == 2 + 8 * 4 + 2
    # chunks of 8192: the second one of 10000 births holds 1808
    assert _count(10_000, overlap=0) == 2 + 6 + 5 + 2
    assert _count(100, overlap=0) == 2 + 5 + 2


def test_time_segments():
    assert _count(1_000_000, overlap=1) == 2 + 8 * 6 + 2
    assert _count(2000, overlap=1) == 2 + 8 * 5 + 2
    assert _count(2000, overlap=1, esc_precision=2) == 2 + 8 * 4 + 2


def test_fp64_step():
    assert bench.launches_per_step(1_000_000, 88256, 1000, 0, True, short=2432) == 4
