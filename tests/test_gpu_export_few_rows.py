"""Exports into outputs of far fewer rows than the graph has vertices: refused with
the number of vertices, and in less time than the export itself (the vertices
are counted by bins, which are not to be so few that the counting waits)."""

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


def outputs(rows, k):
    import torch
    return (torch.zeros((rows, 2) if k > 32 else (rows,), dtype=torch.int64, device="cuda"),
            torch.zeros((rows, 4), dtype=torch.int32, device="cuda"))


def seconds(f):
    import torch
    t = []
    for _ in range(7):
        torch.cuda.synchronize()
        a = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - a)
    return sorted(t)[3]


@pytest.mark.parametrize("k", [31, 51])
@pytest.mark.parametrize("rows", [1, 1000])
def test_a_refused_export_takes_no_longer_than_two(k, rows):
    rs = synth.sample_reads(synth.random_genome(3_000_000, 1), 60_000, 150, 0.002, 1, k, "r")
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    D = len(ref.keys)
    g = dbg.Graph(k, 2 * D)
    g.insert(*to_device(rs))
    all_rows, few = outputs(D, k), outputs(rows, k)

    def refused():
        with pytest.raises(dbg.DbgError) as e:
            g.export_into(*few)
        assert e.value.code == dbg.ERR_BUFFER_TOO_SMALL

    assert seconds(refused) < 2 * seconds(lambda: g.export_into(*all_rows))
    assert np.array_equal(all_rows[0].cpu().numpy().view(np.uint64), ref.keys)
    assert np.array_equal(all_rows[1].cpu().numpy().view(np.uint32), ref.counts)
    g.close()


@pytest.mark.parametrize("k", [21, 51])
def test_a_sixteenth_of_the_table(k):
    # the rows at which the bins turn to the table's size, and outputs that just fit
    rs = synth.ragged_reads(400, 150, k, 3)
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    D = len(ref.keys)
    for slots in (16 * D - 1, 16 * D, 16 * D + 1, 300 * D):
        g = dbg.Graph(k, slots)
        g.insert(*to_device(rs))
        keys, counts = outputs(D, k)
        assert g.export_into(keys, counts) == D
        assert np.array_equal(keys.cpu().numpy().view(np.uint64), ref.keys)
        assert np.array_equal(counts.cpu().numpy().view(np.uint32), ref.counts)
        g.close()


# (12.5 M slots: a warp takes more slots at a time from there on)
@pytest.mark.parametrize("slots", [20_001, 3_000_000, 9_961_471, 9_961_472, 12_500_001])
@pytest.mark.parametrize("k", [25, 51])
def test_sparse_tables(slots, k):
    import torch
    rs = synth.ragged_reads(60, 150, k, 8)
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    D = len(ref.keys)
    g = dbg.Graph(k, slots)
    g.set_tuning(insert_path=1)
    g.insert(*to_device(rs))
    keys, counts = outputs(D, k)
    assert g.export_into(keys, counts) == D
    assert np.array_equal(keys.cpu().numpy().view(np.uint64), ref.keys)
    assert np.array_equal(counts.cpu().numpy().view(np.uint32), ref.counts)
    if k <= 32:  # the caller's scratch, with and without room for a bit per slot
        need = dbg.export_scratch_bytes(k, D, slots)
        for room in (0, slots // 8 + 512):
            keys, counts = outputs(D, k)
            scratch = torch.empty(need + room, dtype=torch.uint8, device="cuda")
            assert g.export_with(keys, counts, scratch) == D
            assert np.array_equal(keys.cpu().numpy().view(np.uint64), ref.keys)
            assert np.array_equal(counts.cpu().numpy().view(np.uint32), ref.counts)
    g.close()


def test_a_sparse_table_is_read_once():
    # 3.2 GB with a few thousand vertices: the export takes about one pass over
    # the table, as counting its vertices does
    rs = synth.ragged_reads(60, 150, 31, 8)
    g = dbg.Graph(31, 100_000_000)
    g.set_tuning(insert_path=1)
    g.insert(*to_device(rs))
    out = outputs(g.stats()[0], 31)
    assert seconds(lambda: g.export_into(*out)) < 1.6 * seconds(g.stats)
    g.close()
