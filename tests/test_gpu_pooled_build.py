"""Rebuilds of mid-size tables through the binned kernels with pooled scratch,
at the sizes where the route changes and in every case that goes back to the
direct insert, against that insert."""

import numpy as np
import pytest

from gpu_util import to_device
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu

POOL_SLOTS = (16 << 20) // 32  # the smallest table that is rebuilt this way
POOL_EVENTS = 4_000_000


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


def reads(n, length, seed, k, genome=60_000):
    return synth.sample_reads(synth.random_genome(genome, seed), n, length, 0.002, seed, k, "r")


def check(g, rs, dev, k, slots, times=1):
    ref = dbg.Graph(k, slots)
    ref.set_tuning(insert_path=1)
    for _ in range(times):
        ref.insert(*dev)
    assert g.status() == ref.status()
    if ref.status() != dbg.OK:  # (a table too small for its reads, on either path)
        ref.close()
        return
    want = ref.export()
    got = g.export()
    assert g.stats() == ref.stats()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    ref.close()


# reserved events just below and at the rule, then more events than reserved
@pytest.mark.parametrize("reserve", [3_200_000, 3_300_000, 300_000_000])
@pytest.mark.parametrize("k,slots", [(21, POOL_SLOTS - 1), (21, POOL_SLOTS), (31, POOL_SLOTS + 12_345),
                                     (31, (256 << 20) // 32 - 1)])
def test_reserved(k, slots, reserve):
    dirty, rs = reads(500, 200, 1, k), reads(40_000, 150, 2, k)
    dev = to_device(rs)
    g = dbg.Graph(k, slots)
    g.insert(*to_device(dirty))
    g.reserve_events(reserve)
    for _ in range(2):  # over the first graph, then over its own
        g.build(*dev)
        check(g, rs, dev, k, slots)
    g.insert(*dev)
    check(g, rs, dev, k, slots, times=2)
    g.close()


# (65,000 reads of 400: more events than the scratch holds, and more vertices than
# the smaller table)
@pytest.mark.parametrize("n,length,slots", [(62_499, 60, 700_000), (62_500, 60, 700_000),
                                            (70_001, 150, 700_000), (65_000, 400, 700_000),
                                            (65_000, 400, 2_500_000)])
def test_by_reads(n, length, slots):
    k = 25
    rs = reads(n, length, 3, k, 30_000)
    dev = to_device(rs)
    g = dbg.Graph(k, slots)
    g.build(*dev)
    check(g, rs, dev, k, slots)
    g.build_host(rs.packed, rs.offsets)
    check(g, rs, dev, k, slots)
    g.close()


def test_a_capture_takes_the_direct_insert():
    import torch
    k, slots = 21, 700_000
    rs = reads(40_000, 150, 5, k)
    dev = to_device(rs)
    g = dbg.Graph(k, slots)
    g.reserve_events(5_000_000)
    torch.cuda.synchronize()
    held = dbg.scratch_bytes()
    s = torch.cuda.Stream()
    cg = torch.cuda.CUDAGraph()
    with torch.cuda.graph(cg, stream=s):
        g.build(*dev, stream=s)
    assert dbg.scratch_bytes() == held
    for _ in range(2):
        cg.replay()
        torch.cuda.synchronize()
        check(g, rs, dev, k, slots)
    g.close()


def test_a_table_too_small_keeps_its_status():
    rs = reads(40_000, 150, 6, 31, 600_000)  # more vertices than slots
    g = dbg.Graph(31, POOL_SLOTS, max_probes=64)
    g.reserve_events(5_000_000)
    dev = to_device(rs)
    g.build(*dev)
    assert g.status() == dbg.ERR_CAPACITY
    few = reads(100, 150, 7, 31)
    g.build(*to_device(few))
    check(g, few, to_device(few), 31, POOL_SLOTS)
    g.close()


def test_two_streams_share_the_pool():
    import torch
    k, slots = 21, 700_000
    sets = [reads(40_000, 150, 8 + i, k) for i in range(4)]
    devs = [to_device(rs) for rs in sets]
    streams = [torch.cuda.Stream() for _ in sets]
    graphs = [dbg.Graph(k, slots) for _ in sets]
    for g in graphs:
        g.reserve_events(5_000_000)
    torch.cuda.synchronize()
    for _ in range(3):
        for g, dev, s in zip(graphs, devs, streams):
            g.build(*dev, stream=s)
    torch.cuda.synchronize()
    for g, rs, dev in zip(graphs, sets, devs):
        check(g, rs, dev, k, slots)
        g.close()
    dbg.release_scratch()
