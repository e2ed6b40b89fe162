"""Events that the global pass finishes: tables so full that probes leave their
tiles and wrap past the table's end, probe limits around the look-ahead of eight
slots, one region and several, against the direct insert."""

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


@pytest.fixture(scope="module", params=[40_000, 400_000])
def sample(request):
    genome = request.param
    rs = synth.sample_reads(synth.random_genome(genome, 5), genome // 30, 150, 0.002, 5, 31, "full")
    dev = to_device(rs)
    g = dbg.Graph(31, 8 * genome)
    g.set_tuning(insert_path=1)
    g.insert(*dev)
    ref = g.export()
    g.close()
    return dev, ref


# (0 free slots: every probe of an absent key may go round the whole table)
@pytest.mark.parametrize("free", [0, 1, 0.02])
def test_full_tables(sample, free):
    dev, (keys, counts) = sample
    D = keys.size
    slots = D + free if isinstance(free, int) else int(D / (1 - free))
    g = dbg.Graph(31, slots, max_probes=slots)
    g.set_tuning(insert_path=2)
    for call, times in ((g.build, 1), (g.insert, 2)):
        call(*dev)
        assert g.status() == dbg.OK
        got = g.export()
        assert np.array_equal(got[0], keys) and np.array_equal(got[1], times * counts)
        assert g.stats() == (D, times * int(counts.astype(np.int64).sum()))
    assert g.binned_counters()["deferred"] > 0
    g.close()


@pytest.mark.parametrize("max_probes", [1, 7, 8, 9, 64])
def test_probe_limits_spill_what_finds_no_slot(sample, max_probes):
    dev, (keys, counts) = sample
    g = dbg.Graph(31, int(keys.size / 0.95), max_probes=max_probes)
    g.set_tuning(insert_path=2)
    g.set_spill(12 * keys.size)
    g.build(*dev)
    assert g.status() == dbg.ERR_NEEDS_GROW
    factor = 8  # (a grown table keeps its probe limit: the shorter, the larger it must be)
    while g.status() == dbg.ERR_NEEDS_GROW and factor <= 128:
        try:
            g.grow(factor * keys.size)
        except dbg.DbgError as e:
            assert e.code == dbg.ERR_CAPACITY
            factor *= 4
    if max_probes == 1:  # (no table holds this many keys without a collision)
        assert g.status() == dbg.ERR_NEEDS_GROW
    else:
        got = g.export()
        assert np.array_equal(got[0], keys) and np.array_equal(got[1], counts)
    g.close()
