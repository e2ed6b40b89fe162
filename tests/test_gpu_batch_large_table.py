"""One large table among many small ones in a batched call: the region size that
suits the average table would cut the large one into more regions than a chain
holds (2,048)."""

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


@pytest.mark.parametrize("at", [0, 150, 299])  # the large table's place in the call
def test_one_large_table_among_small_ones(at):
    rs = synth.sample_reads(synth.random_genome(4_000, 1), 300, 120, 0.0, 1, 31, "r")
    dev = to_device(rs)
    ref = dbg.Graph(31, 10_000)
    ref.set_tuning(insert_path=1)
    ref.insert(*dev)
    keys, counts = ref.export()
    graphs = [dbg.Graph(31, 560_000_000 if i == at else 10_000) for i in range(300)]
    for g in graphs:
        g.reserve_events(50_000)
    items = [(g,) + dev for g in graphs]
    dbg.build_batch(items)
    dbg.insert_batch(items)
    for i in {0, 1, at, 298, 299}:
        got = graphs[i].export()
        assert np.array_equal(got[0], keys) and np.array_equal(got[1], 2 * counts)
    for g in graphs:
        g.close()
    dbg.release_scratch()
