"""Batched inserts into held graphs whose tiles get few and many events: the same
graph as inserted one by one, and for many events a tile in little more time
than the rebuild of the same graphs takes."""

import time

import numpy as np
import pytest

import oracle
from gpu_util import to_device
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


# events a tile (2,048 slots) below and above the 4,096 a CTA loads at a time
@pytest.mark.parametrize("reads,slots", [(2000, 200_000), (17_000, 900_000), (30_000, 500_000)])
def test_few_and_many_events(reads, slots):
    rs = synth.sample_reads(synth.random_genome(30_000, 1), reads + 500, 150, 0.002, 1, 31, "r")
    packed, offsets = to_device(rs)
    g = dbg.Graph(31, slots)
    g.set_tuning(insert_path=2, region_log2=18)
    g.build(packed, offsets[:501])
    g.insert(packed, offsets[500:].clone())
    ref = oracle.build_graph(rs.packed, rs.offsets, 31)
    keys, counts = g.export()
    assert np.array_equal(keys, ref.keys) and np.array_equal(counts, ref.counts)
    g.close()


def seconds(f):
    import torch
    t = []
    for _ in range(9):
        torch.cuda.synchronize()
        a = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - a)
    return sorted(t)[4]


def test_many_events_take_little_more_than_a_rebuild():
    dev = to_device(synth.sample_reads(synth.random_genome(100_000, 1), 13_333, 150, 0.001, 1, 31, "r"))
    graphs = [dbg.Graph(31, 200_000) for _ in range(60)]
    for g in graphs:
        g.reserve_events(1_700_000)
    items = [(g,) + dev for g in graphs]
    rebuild = seconds(lambda: dbg.build_batch(items))
    insert = seconds(lambda: dbg.insert_batch(items))
    assert insert < 1.24 * rebuild, (insert, rebuild)
    for g in graphs:
        g.close()
    dbg.release_scratch()
