"""Calls that have little device memory beside their table: a sparse table of
25.6 GB, everything else but a few hundred megabytes taken."""

import ctypes

import numpy as np
import pytest

import oracle
from gpu_util import to_device
from oracle import contigs as oc
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu

SLOTS = 800_000_000


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


def all_but(megabytes):
    """Device memory taken until about so much is left."""
    import torch
    dbg.release_scratch()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    taken = torch.empty(free - (megabytes << 20), dtype=torch.uint8, device="cuda")
    assert torch.cuda.mem_get_info()[0] <= (megabytes + 4) << 20
    return taken


def graph(rs):
    small = dbg.Graph(rs.k, 100_000)  # (the kernels are loaded before the memory is gone)
    g = dbg.Graph(rs.k, SLOTS)
    dev = to_device(rs)
    for x in (small, g):
        x.set_tuning(insert_path=1)
        x.insert(*dev)
    small.export()
    if rs.k <= 32:
        small.contigs()
    small.close()
    return g


@pytest.mark.parametrize("k", [31, 51])
def test_export_into_more_rows_than_there_is_memory_for(k):
    # (pageable outputs go through temporary ones: 19 GB for a row per slot)
    rs = synth.ragged_reads(300, 150, k, 4)
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    D = len(ref.keys)
    g = graph(rs)
    keys = np.empty((SLOTS, 2) if k > 32 else SLOTS, dtype=np.uint64)  # (pages nobody touches)
    counts = np.empty((SLOTS, 4), dtype=np.uint32)
    taken = all_but(500)
    n = ctypes.c_uint64()
    st = dbg.load().dbg_export_sorted(g.handle, keys.ctypes.data, counts.ctypes.data, SLOTS,
                                      ctypes.byref(n), None)
    assert st == dbg.OK and n.value == D
    assert np.array_equal(keys[:D], ref.keys) and np.array_equal(counts[:D], ref.counts)
    st = dbg.load().dbg_export_sorted(g.handle, None, counts.ctypes.data, D - 1, ctypes.byref(n),
                                      None)
    assert st == dbg.ERR_BUFFER_TOO_SMALL and n.value == D
    del taken
    g.close()
    dbg.release_scratch()


# 1,100 MB: no room for splitters; 500: nor for a list of the usual number of start
# edges; 200: nor for bits of the whole table
@pytest.mark.parametrize("megabytes", [3000, 1100, 500, 200])
def test_contigs(megabytes):
    rs = synth.ragged_reads(300, 150, 31, 4)
    ref = oracle.build_graph(rs.packed, rs.offsets, 31)
    want = oc.find_contigs(ref.keys, ref.counts, 31)
    g = graph(rs)
    taken = all_but(megabytes)
    got = g.contigs()
    del taken
    g.close()
    dbg.release_scratch()
    assert got == want


def test_many_contigs():
    # more memory for the contigs than for anything else: their lists and their
    # text fit, what makes finding them faster does not
    slots = 80_000_000
    rs = synth.sample_reads(synth.random_genome(2_000_000, 2), 2_000_000, 100, 0.02, 2, 21, "r")
    g = dbg.Graph(21, slots)
    g.set_tuning(insert_path=1)
    g.insert(*to_device(rs))
    want = g.contigs()
    S, B = len(want), sum(map(len, want))
    need = slots // 32 * 12 + 64 * S + B
    assert 32 * S > need // 8 + (64 << 20)
    taken = all_but((need + need // 8 + (64 << 20)) >> 20)
    got = g.contigs()
    del taken
    g.close()
    dbg.release_scratch()
    assert got == want
