"""Rebuilds with k from 33 to 63 on the binned path (16-byte events), vertex for
vertex against the oracle: key widths, table loads, region and tile edges,
reads longer than the staging window, keys of all ones, heavy repeats and the
direct fall-back."""

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


def check(g, rs, ref=None):
    ref = ref or oracle.build_graph(rs.packed, rs.offsets, rs.k)
    assert g.status() == dbg.OK
    keys, counts = g.export()
    assert np.array_equal(keys, ref.keys) and np.array_equal(counts, ref.counts)
    assert g.stats() == (len(ref.keys), int(ref.counts.astype(np.int64).sum()))


def vertices(rs):
    return len(oracle.build_graph(rs.packed, rs.offsets, rs.k).keys)


@pytest.mark.parametrize("k", [33, 34, 51, 62, 63, 64])
@pytest.mark.parametrize("lead", [0, 3])
def test_key_widths(k, lead):
    rs = synth.ragged_reads(4000, 220, k, 900 + k, lead=lead)
    g = dbg.Graph(k, int(1.5 * vertices(rs)))
    g.set_tuning(insert_path=2, region_log2=16)
    packed, offsets = to_device(rs, shift=lead)  # (also bytes that are not 16-byte aligned)
    for _ in range(2):  # over a dirty table the second time
        g.build(packed, offsets)
        check(g, rs)
    assert g.binned_counters()["binned"] == (k < 64)
    g.insert(packed, offsets)  # the direct insert adds to the rebuilt table
    keys, counts = g.export()
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    assert np.array_equal(keys, ref.keys) and np.array_equal(counts, 2 * ref.counts)
    g.close()


@pytest.mark.parametrize("slots_over", [0, 1, 2047, 2049, 70_000])
def test_full_tables_and_odd_sizes(slots_over):
    # a load of one with slots_over = 0: probes leave their tiles and wrap
    rs = synth.ragged_reads(3000, 160, 51, 17)
    g = dbg.Graph(51, vertices(rs) + slots_over, max_probes=1 << 30)
    g.set_tuning(insert_path=2, region_log2=16)
    g.build(*to_device(rs))
    check(g, rs)
    g.close()


def test_probe_limit_is_reported():
    rs = synth.ragged_reads(3000, 160, 51, 17)
    g = dbg.Graph(51, vertices(rs) // 2, max_probes=40)
    g.set_tuning(insert_path=2)
    g.build(*to_device(rs))
    assert g.status() == dbg.ERR_CAPACITY
    tiny = synth.from_strings(["ACGT" * 20], 51)
    g.build(*to_device(tiny))
    check(g, tiny)
    g.close()


@pytest.mark.parametrize("k", [33, 51, 63])
def test_long_reads_and_keys_of_all_ones(k):
    text = synth.codes_to_ascii(synth.random_genome(300_000, 6))
    reads = [text[:150_000], "T" * 400, "A" * 300, text[100_000:300_000], "", "ACG", "T" * k, "A" * k]
    rs = synth.from_strings(reads, k, lead=2)
    g = dbg.Graph(k, int(1.5 * vertices(rs)))
    g.set_tuning(insert_path=2)
    g.build(*to_device(rs))
    check(g, rs)
    g.close()


@pytest.mark.parametrize("copies", [300, 20_000])
def test_heavy_repeats(copies):
    # 300: tiles overflow their buckets; 20,000: a region bucket does, and the
    # direct insert takes the call
    base = synth.ragged_reads(4000, 200, 51, 21)
    read = synth.codes_to_ascii(synth.random_genome(150, 8))
    rs = synth.from_strings([base.read_ascii(i) for i in range(base.n_reads)] + [read] * copies, 51)
    g = dbg.Graph(51, 2 * vertices(rs))
    g.set_tuning(insert_path=2, region_log2=16)
    g.build(*to_device(rs))
    check(g, rs)
    g.close()


def test_host_input_batch_and_automatic_path():
    rs = synth.sample_reads(synth.random_genome(40_000, 3), 6000, 130, 0.01, 3, 51, "w")
    ref = oracle.build_graph(rs.packed, rs.offsets, 51)
    g = dbg.Graph(51, 8_500_000)  # over 256 MiB: binned without being asked
    g.build_host(rs.packed, rs.offsets)
    check(g, rs, ref)
    assert g.binned_counters()["binned"]
    narrow = synth.ragged_reads(500, 100, 21, 4)
    h = dbg.Graph(21, 100_000)
    items = [(g,) + to_device(rs), (h,) + to_device(narrow)]
    dbg.build_batch(items)
    check(g, rs, ref)
    nref = oracle.build_graph(narrow.packed, narrow.offsets, 21)
    assert np.array_equal(h.export()[0], nref.keys)
    for x in (g, h):
        x.close()


def test_captured_rebuild():
    import torch
    rs = synth.ragged_reads(2000, 160, 51, 33)
    ref = oracle.build_graph(rs.packed, rs.offsets, 51)
    packed, offsets = to_device(rs)
    for warm in (False, True):  # without its scratch the capture takes the direct insert
        g = dbg.Graph(51, 2 * len(ref.keys))
        g.set_tuning(insert_path=2)
        if warm:
            g.build(packed, offsets)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            g.build(packed, offsets)
        for _ in range(2):
            graph.replay()
        torch.cuda.synchronize()
        check(g, rs, ref)
        g.close()


def test_decreasing_offsets_are_reported():
    import torch
    rs = synth.ragged_reads(600, 160, 51, 41)
    packed, offsets = to_device(rs)
    for at in (300, 600):
        bad = offsets.clone()
        bad[at:] = 0
        g = dbg.Graph(51, 100_000)
        g.set_tuning(insert_path=2)
        g.build(packed, bad)
        assert g.status() == dbg.ERR_BAD_OFFSETS
        g.close()
    assert torch.cuda.is_available()
