"""Direct inserts of many reads, whose tiles the device sizes by their length: short
reads, reads shorter than k, very uneven ones, and the read counts around the
rule, against the oracle."""

import numpy as np
import pytest

import oracle
from gpu_util import to_device
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu

ASK = 12 * 152 * 8  # more reads than this: the device is asked


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


@pytest.mark.parametrize("k", [21, 32, 51])
@pytest.mark.parametrize("n,length,every,other", [
    (ASK, 60, 1, 0), (ASK + 1, 60, 1, 0), (ASK + 1, 52, 1, 0), (40_000, 54, 1, 0),
    (40_000, 30, 1, 0), (40_000, 60, 97, 3), (15_000, 60, 3000, 40_000), (60_000, 53, 2, 10)])
def test_short_and_uneven_reads(k, n, length, every, other):
    # `every`-th reads have `other` bases
    text = synth.codes_to_ascii(synth.random_genome(80_000, n))
    rng = np.random.default_rng(k + n)
    lens = [other if other and i % every == every - 1 else length for i in range(n)]
    starts = rng.integers(0, 80_000 - 40_000, n)
    rs = synth.from_strings([text[s:s + m] for s, m in zip(starts, lens)], k, lead=n % 3)
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    g = dbg.Graph(k, 2 * len(ref.keys) + 64)
    g.insert(*to_device(rs))
    keys, counts = g.export()
    assert np.array_equal(keys, ref.keys) and np.array_equal(counts, ref.counts)
    g.close()


def test_decreasing_offsets_are_reported():
    rs = synth.sample_reads(synth.random_genome(20_000, 1), ASK + 100, 40, 0.0, 1, 21, "r")
    packed, offsets = to_device(rs)
    for at in (ASK // 2, ASK + 100):  # (a later read, and the last offset itself)
        bad = offsets.clone()
        bad[at:] = 0
        g = dbg.Graph(21, 100_000)
        g.insert(packed, bad)
        assert g.status() == dbg.ERR_BAD_OFFSETS
        g.close()


def test_many_read_sets_in_one_launch():
    sets = [synth.sample_reads(synth.random_genome(3000, i), 700, 40, 0.0, i, 32, "r")
            for i in range(130)]
    graphs = [dbg.Graph(32, 8000) for _ in sets]
    dbg.build_batch([(g,) + to_device(rs) for g, rs in zip(graphs, sets)])
    for g, rs in list(zip(graphs, sets))[::13]:
        ref = oracle.build_graph(rs.packed, rs.offsets, 32)
        keys, counts = g.export()
        assert np.array_equal(keys, ref.keys) and np.array_equal(counts, ref.counts)
    for g in graphs:
        g.close()
