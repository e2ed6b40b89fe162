"""The sorted export of graphs whose keys crowd into some bins: genomes of uneven
base composition, low-complexity stretches and reads that share their first
bases, from records, in place, to pinned memory and with the caller's scratch,
against the oracle."""

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


def text(rng, n, gc):
    p = [(1 - gc) / 2, gc / 2, gc / 2, (1 - gc) / 2]
    return synth.codes_to_ascii(rng.choice(4, n, p=p).astype(np.uint8))


def shared_start(rng, k, shared, n):
    """n reads of k bases that begin with the same `shared`."""
    head = synth.codes_to_ascii(rng.integers(0, 4, shared).astype(np.uint8))
    return [head + synth.codes_to_ascii(rng.integers(0, 4, k - shared).astype(np.uint8))
            for _ in range(n)]


def rows_of(keys, counts, n):
    import torch
    if isinstance(keys, torch.Tensor):
        keys, counts = keys.cpu().numpy(), counts.cpu().numpy()
    return keys[:n].view(np.uint64), counts[:n].view(np.uint32)


def check(rs, k, rows_over=0):
    import torch
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    D = len(ref.keys)
    dev = to_device(rs)

    def outputs(**where):
        rows = D + rows_over
        return (torch.full((rows, 2) if k > 32 else (rows,), -7, dtype=torch.int64, **where),
                torch.full((rows, 4), -7, dtype=torch.int32, **where))

    def same(keys, counts):
        got = rows_of(keys, counts, D)
        assert np.array_equal(got[0], ref.keys) and np.array_equal(got[1], ref.counts)
        assert bool((keys[D:] == -7).all()) and bool((counts[D:] == -7).all())

    for path in (1, 2):  # in place (k <= 32), or records in the event buffer
        g = dbg.Graph(k, 2 * D + 64)
        g.set_tuning(insert_path=path)
        g.build(*dev)
        out = outputs(device="cuda")
        assert g.export_into(*out) == D
        same(*out)
        keys, counts = outputs(pin_memory=True)
        got = g.export(out=(keys.numpy(), counts.numpy()))
        assert len(got[0]) == D
        same(keys, counts)
        got = g.export()
        assert np.array_equal(got[0], ref.keys) and np.array_equal(got[1], ref.counts)
        if k <= 32:
            need = dbg.export_scratch_bytes(k, D, g.info()["n_slots"])
            for extra in (0, 64 * D):  # (room for the crowded records beside the bins, or not)
                scratch = torch.empty(need + extra, dtype=torch.uint8, device="cuda")
                out = outputs(device="cuda")
                assert g.export_with(*out, scratch) == D
                got = rows_of(*out, D)
                assert np.array_equal(got[0], ref.keys) and np.array_equal(got[1], ref.counts)
        g.close()


@pytest.mark.parametrize("k", [21, 31, 32, 33, 51])
@pytest.mark.parametrize("gc", [0.35, 0.2, 0.1])
def test_uneven_bases(k, gc):
    rng = np.random.default_rng(k)
    genome = text(rng, 400_000, gc)
    starts = rng.integers(0, 400_000 - 150, 6000)
    check(synth.from_strings([genome[i:i + 150] for i in starts], k), k)


# bins of one record less than a bucket can take beside the others, of as many, and
# far more; few records besides, so that buckets are small, and many
@pytest.mark.parametrize("k,shared", [(31, 14), (33, 20), (51, 20)])
@pytest.mark.parametrize("n", [1000, 1900, 1930, 2048, 2049, 6000, 30_000])
@pytest.mark.parametrize("others", [20_000, 500_000])
def test_a_bin_above_the_cap(k, shared, n, others):
    rng = np.random.default_rng(n + k)
    reads = shared_start(rng, k, shared, n)
    check(synth.from_strings(reads + [text(rng, others, 0.5)], k), k, rows_over=3)


@pytest.mark.parametrize("k", [31, 51])
def test_several_crowded_buckets_at_both_ends(k):
    rng = np.random.default_rng(7)
    reads = []
    for base in "ACGT":  # (the first and the last keys among them)
        reads += [base * (k // 2) + synth.codes_to_ascii(rng.integers(0, 4, k - k // 2).astype(np.uint8))
                  for _ in range(3000)]
    reads += ["A" * k, "T" * k, "A" * (k - 1) + "T"]
    check(synth.from_strings(reads + [text(rng, 100_000, 0.5)], k), k)


def sampled(genome, n, length, gc, err, seed):
    """(packed, offsets) of n reads of a genome of that base composition, made on the GPU."""
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    at = (1 - gc) / 2
    edges = torch.tensor([at, 0.5, 1 - at], device="cuda")

    def bases(m):
        return torch.bucketize(torch.rand(m, device="cuda", generator=gen), edges,
                               right=True).to(torch.uint8)

    text = bases(genome)
    starts = torch.randint(0, genome - length + 1, (n, 1), device="cuda", generator=gen)
    reads = text[starts + torch.arange(length, device="cuda")].view(-1)
    wrong = torch.rand(reads.numel(), device="cuda", generator=gen) < err
    reads = torch.where(wrong, bases(reads.numel()), reads).view(-1, 4)
    packed = reads[:, 0] | (reads[:, 1] << 2) | (reads[:, 2] << 4) | (reads[:, 3] << 6)
    return packed, torch.arange(n + 1, device="cuda") * length


def test_uneven_bases_take_little_longer():
    # about 20 M vertices of 126 bits: a radix sort of all takes some four times as long
    import time
    import torch
    k, took = 64, {}
    for gc in (0.5, 0.2):
        packed, offsets = sampled(2_000_000, 400_000, 152, gc, 0.01, 5)
        g = dbg.Graph(k, 45_000_000)
        g.build(packed, offsets)
        D = g.stats()[0]
        keys = torch.zeros((D, 2), dtype=torch.int64, device="cuda")
        counts = torch.zeros((D, 4), dtype=torch.int32, device="cuda")
        t = []
        for _ in range(5):
            torch.cuda.synchronize()
            a = time.perf_counter()
            assert g.export_into(keys, counts) == D
            torch.cuda.synchronize()
            t.append(time.perf_counter() - a)
        took[gc] = sorted(t)[2] / D
        hi, lo = keys[:, 0], keys[:, 1] ^ (-1 << 63)  # (the high words are positive)
        assert bool(((hi[1:] > hi[:-1]) | ((hi[1:] == hi[:-1]) & (lo[1:] > lo[:-1]))).all())
        assert int(counts.sum(dtype=torch.int64)) == g.stats()[1]
        g.close()
        del packed, offsets, keys, counts
    assert took[0.2] < 2 * took[0.5], took
