"""The binned scatter's tiles for read sets of one read to more than a whole wave
of tiles, long and short, against the direct insert."""

import numpy as np
import pytest

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


# the scatter's tiles: one read to past the last whole wave, long and short reads
@pytest.mark.parametrize("n,length", [(1, 300), (9, 5000), (300, 2500), (2433, 100), (30_000, 90),
                                      (130_000, 40)])
def test_scatter_tiles(n, length):
    k, slots = 21, 1_500_000
    rs = reads(n, length, 11, k)
    dev = to_device(rs)
    g = dbg.Graph(k, slots)
    g.set_tuning(insert_path=2)
    g.build(*dev)
    check(g, rs, dev, k, slots)
    dbg.build_batch([(g, *dev)])
    check(g, rs, dev, k, slots)
    assert n < 2 or g.stats()[0] > 0
    g.close()
