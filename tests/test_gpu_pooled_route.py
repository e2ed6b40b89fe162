"""Which rebuilds of mid-size tables take the binned kernels, as the pool's growth
shows (17 bytes an event of scratch), and that short reads are not among them
before they pay."""

import time

import pytest

from gpu_util import to_device
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu

EVENTS = 8_000_000


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


def reads(n, length, k):
    return to_device(synth.sample_reads(synth.random_genome(60_000, 3), n, length, 0.0, 3, k, "r"))


def pool_growth(g, dev):
    import torch
    torch.cuda.synchronize()
    dbg.release_scratch()
    held = dbg.scratch_bytes()
    g.build(*dev)
    torch.cuda.synchronize()
    return dbg.scratch_bytes() - held


# (dbg_reserve_events adds a sixteenth and about 0.6 M)
@pytest.mark.parametrize("slots,reserve,pooled", [
    (700_000, 9_000_000, True), (700_000, 6_000_000, False), (500_000, 9_000_000, False),
    (1 << 23, 9_000_000, None), ((1 << 23) - 1, 9_000_000, True), (700_000, 200_000_000, False)])
@pytest.mark.parametrize("path", [0, 1])
def test_by_reserved_events_and_table(slots, reserve, pooled, path):
    dev = reads(3000, 100, 21)
    g = dbg.Graph(21, slots)
    g.reserve_events(reserve)
    g.set_tuning(insert_path=path)
    grown = pool_growth(g, dev)
    if path == 1 or not pooled:  # (None: binned with the handle's own buffers)
        assert grown == 0
    else:
        assert grown >= 17 * reserve
        g.enable_kernel_timing(1)
        g.build(*dev)
        times = dict(zip(g.KERNELS, g.kernel_times()[0]))
        assert times["bin_apply"] > times["direct_fallback"] > 0
    g.close()


@pytest.mark.parametrize("n,pooled", [(EVENTS // 8 - 1, False), (EVENTS // 8, True)])
def test_by_reads(n, pooled):
    dev = reads(n, 60, 21)
    g = dbg.Graph(21, 700_000)
    assert (pool_growth(g, dev) >= 17 * EVENTS) == pooled
    g.close()


def seconds(f, before=lambda: None):
    import torch
    t = []
    for _ in range(9):
        before()
        torch.cuda.synchronize()
        a = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - a)
    return sorted(t)[4]


@pytest.mark.parametrize("k,length,n", [(31, 36, 571_000), (21, 50, 133_000), (31, 50, 180_000)])
def test_short_reads_are_not_held_up(k, length, n):
    dev = reads(n, length, k)
    g = dbg.Graph(k, 2_500_000)
    insert = seconds(lambda: g.insert(*dev), g.reset)
    assert seconds(lambda: g.build(*dev)) < 1.15 * insert + 25e-6
    g.close()
