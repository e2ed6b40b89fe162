"""dbg_stats after captured calls are replayed: the host sees a call when it is
captured, the graph changes when it is replayed, and the counts are the
graph's all the same."""

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


def reads(n, seed, k):
    return synth.sample_reads(synth.random_genome(60_000, seed), n, 150, 0.002, seed, k, "r")


def counted(g):
    keys, counts = g.export()
    return len(keys), int(counts.astype(np.int64).sum())


# (21: a table whose rebuild takes pooled scratch, captured calls the direct insert;
# 31 binned and streaming; 51: a wide binned rebuild, a direct insert)
TUNINGS = {"pooled": (21, {}), "binned": (31, dict(insert_path=2)),
           "streaming": (31, dict(insert_path=2, apply_mode=1)), "wide": (51, dict(insert_path=2))}


@pytest.mark.parametrize("call", ["insert", "insert_batch", "reset", "build", "build_batch"])
@pytest.mark.parametrize("form", list(TUNINGS))
def test_a_replayed_call_is_counted(form, call):
    import torch
    k, tuning = TUNINGS[form]
    first, more = reads(3000, 1, k), reads(30_000, 2, k)
    a, b = to_device(first), to_device(more)
    g = dbg.Graph(k, 700_000)
    g.reserve_events(5_000_000)
    calls = {"insert": lambda: g.insert(*a), "reset": g.reset, "build": lambda: g.build(*a),
             "insert_batch": lambda: dbg.insert_batch([(g,) + a]),
             "build_batch": lambda: dbg.build_batch([(g,) + a])}
    if tuning:
        g.set_tuning(**tuning)
    if form != "pooled":
        calls[call]()  # (the buffers a capture cannot make)
    torch.cuda.synchronize()
    cg = torch.cuda.CUDAGraph()
    with torch.cuda.graph(cg):
        calls[call]()
    if form == "streaming":  # the plain rebuild counts, the captured call does not
        g.set_tuning(insert_path=2)
    g.build(*b)
    plain = counted(g)
    assert g.stats() == plain
    cg.replay()
    torch.cuda.synchronize()
    after = counted(g)
    assert after != plain
    assert g.stats() == after
    g.close()


def test_a_rebuild_captured_after_normalize_is_not_counted_before_its_replay():
    import torch
    k = 31
    a = to_device(reads(30_000, 3, k))
    g = dbg.Graph(k, 700_000)
    g.set_tuning(insert_path=2)
    g.build(*a)
    plain = g.stats()
    g.normalize(20.0)
    torch.cuda.synchronize()
    cg = torch.cuda.CUDAGraph()
    with torch.cuda.graph(cg):
        g.build(*a)
    torch.cuda.synchronize()
    assert g.stats() == counted(g) != plain
    cg.replay()
    torch.cuda.synchronize()
    assert g.stats() == plain
    g.close()
