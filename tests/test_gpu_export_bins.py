"""The sorted export by bins at the edges of its buckets and outputs, against
the oracle: small graphs, one- and two-word keys, records in the event buffer
and in place, outputs of more rows than vertices, host and unaligned outputs."""

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


def expected(rs):
    return oracle.build_graph(rs.packed, rs.offsets, rs.k)


def same(keys, counts, ref, n):
    import torch
    if isinstance(keys, torch.Tensor):
        keys, counts = keys.cpu().numpy(), counts.cpu().numpy()
    assert np.array_equal(keys[:n].view(np.uint64), ref.keys)
    assert np.array_equal(counts[:n].view(np.uint32), ref.counts)


def outputs(rows, k, pad=0):
    import torch
    keys = torch.full((rows * (2 if k > 32 else 1) + pad,), -7, dtype=torch.int64, device="cuda")[pad:]
    counts = torch.full((rows * 4 + pad,), -7, dtype=torch.int32, device="cuda")[pad:]
    return keys.view(rows, 2) if k > 32 else keys, counts.view(rows, 4)


# (read length, reads): from one vertex pair up to buckets of every size
@pytest.mark.parametrize("reads", [0, 1, 2, 9, 70, 600, 5000, 30000])
@pytest.mark.parametrize("k", [2, 5, 11, 31, 32, 33, 51, 64])
def test_sizes_and_keys(reads, k):
    rs = synth.ragged_reads(reads, 100, k, 31 * reads + k)
    ref = expected(rs)
    D = len(ref.keys)
    g = dbg.Graph(k, max(64, 2 * D + 16))
    g.insert(*to_device(rs))
    for rows in {max(1, D), D + 1, 3 * D + 5}:
        keys, counts = outputs(rows, k)
        assert g.export_into(keys, counts) == D
        same(keys, counts, ref, D)
    g.close()


@pytest.mark.parametrize("fill", [0.3, 0.95])
@pytest.mark.parametrize("k", [12, 31])
def test_records_in_the_event_buffer(k, fill):
    rs = synth.sample_reads(synth.random_genome(200_000, 5), 20_000, 120, 0.01, 5, k, "bins")
    ref = expected(rs)
    D = len(ref.keys)
    g = dbg.Graph(k, int(D / fill))
    g.set_tuning(insert_path=2, region_log2=16)
    packed, offsets = to_device(rs)
    keys, counts = outputs(D, k)
    for _ in range(2):  # the export's records and the next build share the buffer
        g.build(packed, offsets)
        assert g.export_into(keys, counts) == D
        same(keys, counts, ref, D)
    g.insert(packed, offsets)  # and an insert into the held graph after it
    keys, counts = outputs(D, k)
    assert g.export_into(keys, counts) == D
    assert np.array_equal(counts.cpu().numpy().view(np.uint32), 2 * ref.counts)
    g.close()


@pytest.mark.parametrize("k", [31, 51])
def test_host_unaligned_and_single_outputs(k):
    rs = synth.ragged_reads(3000, 150, k, 77)
    ref = expected(rs)
    D = len(ref.keys)
    g = dbg.Graph(k, 2 * D)
    g.insert(*to_device(rs))
    keys, counts = g.export()
    same(keys, counts, ref, D)
    keys, counts = outputs(D, k, pad=1)  # 8- and 4-byte aligned
    assert g.export_into(keys, counts) == D
    same(keys, counts, ref, D)
    import ctypes
    n = ctypes.c_uint64()
    only = np.zeros((D, 4), dtype=np.uint32)
    L = dbg.load()
    assert L.dbg_export_sorted(g.handle, None, only.ctypes.data, D, ctypes.byref(n), None) == dbg.OK
    assert n.value == D and np.array_equal(only, ref.counts)
    # too few rows: refused, the count told
    keys, counts = outputs(max(1, D // 3), k)
    with pytest.raises(dbg.DbgError) as e:
        g.export_into(keys, counts)
    assert e.value.code == dbg.ERR_BUFFER_TOO_SMALL
    g.close()


@pytest.mark.parametrize("k,shared", [(31, 20), (51, 30)])
@pytest.mark.parametrize("n", [900, 5000])
def test_keys_crowded_into_one_bin(k, shared, n):
    # n reads that share their first bases: one bin of n keys (5,000: more
    # than a bucket holds, left to the radix sort)
    rng = np.random.default_rng(n)
    head = synth.codes_to_ascii(synth.random_genome(shared, 9))
    reads = [head + synth.codes_to_ascii(rng.integers(0, 4, k - shared)) for _ in range(n)]
    rs = synth.from_strings(reads + [synth.codes_to_ascii(synth.random_genome(20_000, 4))], k)
    ref = expected(rs)
    D = len(ref.keys)
    g = dbg.Graph(k, 2 * D)
    g.insert(*to_device(rs))
    keys, counts = outputs(D, k)
    assert g.export_into(keys, counts) == D
    same(keys, counts, ref, D)
    g.close()


@pytest.mark.parametrize("k", [21, 51])
@pytest.mark.parametrize("reads,crowd", [(1, 0), (4000, 0), (300, 5000)])
def test_pinned_host_outputs(k, reads, crowd):
    # written by the sort itself; keys crowded into one bin go the copied way
    import torch
    rng = np.random.default_rng(k)
    head = synth.codes_to_ascii(synth.random_genome(k // 2, 9))
    base = synth.ragged_reads(reads, 120, k, 5)
    texts = [head + synth.codes_to_ascii(rng.integers(0, 4, k - k // 2)) for _ in range(crowd)]
    rs = synth.from_strings(texts + [base.read_ascii(i) for i in range(reads)] + ["ACGT" * 30], k)
    ref = expected(rs)
    D = len(ref.keys)
    g = dbg.Graph(k, 2 * D + 8)
    g.insert(*to_device(rs))
    for rows in (D, 2 * D + 3):
        keys = torch.full((rows, 2) if k > 32 else (rows,), -7, dtype=torch.int64, pin_memory=True)
        counts = torch.full((rows, 4), -7, dtype=torch.int32, pin_memory=True)
        got = g.export(out=(keys.numpy(), counts.numpy()))
        assert len(got[0]) == D
        same(keys, counts, ref, D)
        assert bool((keys[D:] == -7).all()) and bool((counts[D:] == -7).all())
    keys = torch.full((1, 2) if k > 32 else (1,), -7, dtype=torch.int64, pin_memory=True)
    counts = torch.full((1, 4), -7, dtype=torch.int32, pin_memory=True)
    import ctypes
    n = ctypes.c_uint64()
    st = dbg.load().dbg_export_sorted(g.handle, keys.data_ptr(), counts.data_ptr(), 1,
                                      ctypes.byref(n), None)
    assert st == dbg.ERR_BUFFER_TOO_SMALL and n.value == D and bool((keys == -7).all())
    g.close()


@pytest.mark.parametrize("k", [11, 31])
@pytest.mark.parametrize("reads", [1, 400, 30_000])
def test_large_outputs_placed_by_bucket(k, reads):
    # a direct insert has no event buffer to sort records in; above 2^21 rows
    # the keys and rows are placed by their bucket
    rs = synth.ragged_reads(reads, 160, k, 13 * reads + k)
    ref = expected(rs)
    D = len(ref.keys)
    rows = (1 << 21) + 4099
    g = dbg.Graph(k, rows)
    g.set_tuning(insert_path=1)
    g.insert(*to_device(rs))
    keys, counts = outputs(rows, k)
    assert g.export_into(keys, counts) == D
    same(keys, counts, ref, D)
    assert bool((keys[D:] == -7).all()) and bool((counts[D:] == -7).all())
    g.close()
