"""The scratch of rebuilds with k > 32 belongs to the library: graphs share it, it is
counted and given back, and a graph that finds no memory gets it."""

import threading

import numpy as np
import pytest

import oracle
from gpu_util import to_device
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu

K, SLOTS = 51, 9_000_000  # over 256 MiB: binned without being asked


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


@pytest.fixture(autouse=True)
def _nothing_held():
    dbg.release_scratch()
    yield
    dbg.release_scratch()


def reads(seed):
    rs = synth.sample_reads(synth.random_genome(30_000, seed), 4000, 130, 0.01, seed, K, "w")
    return to_device(rs), oracle.build_graph(rs.packed, rs.offsets, K)


def check(g, ref, stream=None):
    keys, counts = g.export(stream=stream)
    assert np.array_equal(keys, ref.keys) and np.array_equal(counts, ref.counts)


def test_graphs_share_one_scratch_that_is_given_back():
    sets = [reads(i) for i in range(3)]
    graphs = [dbg.Graph(K, SLOTS + 1000 * i) for i in range(3)]
    held = []
    for g, (dev, ref) in zip(graphs, sets):
        g.build(*dev)
        check(g, ref)
        assert g.binned_counters()["binned"]
        held.append(dbg.scratch_bytes())
    assert held[0] > 34 * 3 * SLOTS  # (16-byte events, two buffers, three events a slot)
    assert held[2] - held[0] < 64 << 20  # (the larger tables' rest, and the exports' pool)
    dbg.release_scratch()
    assert dbg.scratch_bytes() == 0
    for g, (dev, ref) in zip(graphs, sets):
        check(g, ref)  # (the graphs are whole without it)
        g.build(*dev)
        check(g, ref)
        told = g.binned_counters()
        g.insert(*dev)
        assert told["binned"] and g.binned_counters() == told
        g.close()


def test_a_graph_finds_the_memory_that_the_scratch_holds():
    import torch
    dev, ref = reads(5)
    g = dbg.Graph(K, SLOTS)
    g.build(*dev)
    g.export()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = dbg.scratch_bytes()
    free = torch.cuda.mem_get_info()[0]
    taken = torch.empty(free - (64 << 20), dtype=torch.uint8, device="cuda")
    more = dbg.Graph(31, held // 2 // 32)  # (half of it)
    assert dbg.scratch_bytes() < held
    more.close()
    g.build(*dev)  # (and without memory for its scratch the direct insert does it)
    del taken
    check(g, ref)
    g.close()


def test_streams_and_threads():
    import torch
    sets = [reads(10 + i) for i in range(4)]
    graphs = [dbg.Graph(K, SLOTS + 50_000 * i) for i in range(4)]
    torch.cuda.synchronize()
    wrong = []

    def work(i):
        s = torch.cuda.Stream()
        for again in range(4):
            dev, ref = sets[(i + again) % 4]
            graphs[i].build(*dev, stream=s)
            keys, counts = graphs[i].export(stream=s)
            if not (np.array_equal(keys, ref.keys) and np.array_equal(counts, ref.counts)):
                wrong.append((i, again))
            if i == 0 and again == 1:
                dbg.release_scratch()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    for g in graphs:
        g.close()


def test_a_captured_rebuild_outlives_the_scratch():
    import torch
    dev, ref = reads(20)
    g = dbg.Graph(K, SLOTS)
    g.build(*dev)
    torch.cuda.synchronize()
    cg = torch.cuda.CUDAGraph()
    with torch.cuda.graph(cg):
        g.build(*dev)
    dbg.release_scratch()
    g.insert(*dev)
    cg.replay()
    torch.cuda.synchronize()
    check(g, ref)
    g.close()
