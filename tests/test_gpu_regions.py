"""Table sizes at the edges of the automatic region rule (2^18 slots at least,
256 regions a table, 1,024 a chain of tables), rebuilt over a dirty table and
inserted into a held one, against the direct insert of the same reads."""

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


def reads(seed):
    return synth.sample_reads(synth.random_genome(60_000, seed), 8_000, 120, 0.01, seed, 31, "r")


def direct(rs):
    g = dbg.Graph(31, 1_500_000)
    g.set_tuning(insert_path=1)
    g.insert(*to_device(rs))
    out = g.export()
    g.close()
    return out


@pytest.mark.parametrize("slots", [(1 << 18) - 1, (1 << 18) + 1, 256 * (1 << 18), 256 * (1 << 18) + 1])
def test_one_table(slots):
    first, second = reads(1), reads(2)
    g = dbg.Graph(31, slots)
    g.set_tuning(insert_path=2)
    g.build(*to_device(first))
    g.build(*to_device(second))  # over the first graph, whose status and counts it drops
    keys, counts = direct(second)
    got = g.export()
    assert np.array_equal(got[0], keys) and np.array_equal(got[1], counts)
    assert g.stats() == (keys.size, int(counts.astype(np.int64).sum()))
    assert g.binned_counters()["binned"]
    g.insert(*to_device(second))
    got = g.export()
    assert np.array_equal(got[0], keys) and np.array_equal(got[1], 2 * counts)
    g.close()


@pytest.mark.parametrize("tables,slots", [(3, 1 << 18), (5, 55_000_000), (130, 300_001)])
def test_chain_of_tables(tables, slots):
    sets = [reads(10 + i % 4) for i in range(tables)]
    refs = {i: direct(reads(10 + i)) for i in range(4)}
    graphs = [dbg.Graph(31, slots) for _ in sets]
    items = [(g,) + to_device(rs) for g, rs in zip(graphs, sets)]
    for _ in range(2):
        dbg.build_batch(items)
    for i, g in enumerate(graphs):
        got = g.export()
        assert np.array_equal(got[0], refs[i % 4][0]) and np.array_equal(got[1], refs[i % 4][1])
        g.close()
    dbg.release_scratch()


def test_a_failed_build_is_cleared_by_the_next():
    small = reads(3)
    g = dbg.Graph(31, 2000, max_probes=64)  # far too small: the sticky status is set
    g.build(*to_device(small))
    assert g.status() == dbg.ERR_CAPACITY
    tiny = synth.from_strings(["ACGT" * 12], 31)
    for path in (1, 2):
        g.set_tuning(insert_path=path)
        g.build(*to_device(small))
        assert g.status() == dbg.ERR_CAPACITY
        g.build(*to_device(tiny))
        assert g.status() == dbg.OK and g.stats()[1] == tiny.n_edges()
    g.build(*to_device(small))
    g.reset()
    assert g.status() == dbg.OK and g.stats() == (0, 0)
    g.close()


@pytest.mark.parametrize("slots_over", [0, 3, 5000])
@pytest.mark.parametrize("max_probes", [0, 1 << 30])
def test_probes_that_leave_their_tile(slots_over, max_probes):
    # tables at a load near one: many events are applied past their tile's end,
    # and wrap past the table's
    rs = reads(7)
    keys, counts = direct(rs)
    g = dbg.Graph(31, keys.size + slots_over, max_probes=max_probes)
    g.set_tuning(insert_path=2, region_log2=16)
    g.set_spill(100_000)
    g.build(*to_device(rs))
    if g.status() == dbg.ERR_NEEDS_GROW:
        g.grow(2 * keys.size)
    got = g.export()
    assert np.array_equal(got[0], keys) and np.array_equal(got[1], counts)
    g.close()
