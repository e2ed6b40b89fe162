"""Contigs long enough to be cut at splitters, shared tails and cycles, string
for string against the oracle; normalization past the table of small counts."""

import numpy as np
import pytest

import oracle
from gpu_util import gpu_graph
from oracle import contigs as oc
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


def random_text(n, seed):
    return synth.codes_to_ascii(synth.random_genome(n, seed))


def check(reads, k):
    rs = synth.from_strings(reads, k)
    g = gpu_graph(rs)
    got = g.contigs()
    g.close()
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    assert got == oc.find_contigs(ref.keys, ref.counts, k)
    return got


@pytest.mark.parametrize("length", [40, 400, 30_000])
def test_one_long_contig(length):
    text = random_text(length, length)
    assert check([text], 21) == [text]


@pytest.mark.parametrize("cycle", [1, 3, 40, 700, 5000])
@pytest.mark.parametrize("tail", [25, 3000])
def test_tail_into_cycle(cycle, tail):
    k = 21
    loop = random_text(cycle, 7 + cycle)
    loop = (loop * (k // cycle + 2))[:cycle + k] if cycle < k else loop + loop[:k]
    got = check([random_text(tail, 11) + loop], k)
    assert len(got) == 1 and len(got[0]) >= tail + min(cycle, k - 1)


def test_many_contigs_share_a_long_tail():
    # more jumps in all than the first guess of the unit list holds
    tail = random_text(12_000, 3)
    reads = [random_text(60, 100 + i) + tail for i in range(200)]
    got = check(reads, 21)
    assert len(got) == 200 and all(len(c) == 12_060 for c in got)


@pytest.mark.parametrize("divisor", [1.0, 3.0, 700.0])
def test_normalize_small_and_large_counts(divisor):
    # counts of 1, 7, 1023, 1024, 1500: below, at and past the table of quotients
    reads = [r for i, n in enumerate((1, 7, 1023, 1024, 1500)) for r in [random_text(30, 50 + i)] * n]
    rs = synth.from_strings(reads, 21)
    ref = oracle.build_graph(rs.packed, rs.offsets, 21)
    g = gpu_graph(rs)
    g.normalize(divisor)
    keys, counts = g.export()
    g.close()
    assert np.array_equal(keys, ref.keys)
    assert np.array_equal(counts, oc.normalize(ref.counts, divisor))


# (tables at the edges of the splitters' spacings and of the room for more levels)
@pytest.mark.parametrize("slots", [1 << 20, (1 << 20) + 1, (1 << 21) + 1, (1 << 22) + 1, 1 << 23,
                                   (1 << 23) + 1])
def test_table_sizes(slots):
    k = 21
    tail = random_text(9_000, 3)
    loop = random_text(3000, 8)
    texts = [random_text(n, 200 + n) for n in (25, 700, 250_000)]
    texts += [random_text(60, 100 + i) + tail for i in range(20)] + [random_text(500, 9) + loop + loop[:k]]
    rs = synth.from_strings(texts, k)
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    g = gpu_graph(rs, capacity=slots)
    assert g.contigs() == oc.find_contigs(ref.keys, ref.counts, k)
    g.close()
