"""Results that kernels report to pinned memory: more calls at once than there are
slots, and calls after the page was given back, which copy them instead."""

import threading

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


@pytest.mark.parametrize("threads", [1, 90])
def test_calls_at_once(threads):
    import torch
    sets = [synth.ragged_reads(40 + i, 120, 21, 900 + i) for i in range(threads)]
    want = []
    graphs = []
    for rs in sets:
        g = dbg.Graph(21, 20_000)
        g.build(*to_device(rs))
        want.append((g.stats(), g.export(), g.contigs()))
        graphs.append(g)
    dbg.release_scratch()  # (and the page with it: copied from here on, until a graph is made)
    for again in range(2):
        wrong = []

        def work(i):
            s = torch.cuda.Stream()
            g = graphs[i]
            for _ in range(3):
                k, c = g.export(stream=s)
                if (g.stats(stream=s) != want[i][0] or g.status(stream=s) != dbg.OK or
                        not np.array_equal(k, want[i][1][0]) or
                        not np.array_equal(c, want[i][1][1]) or
                        g.contigs(stream=s) != want[i][2]):
                    wrong.append(i)

        ts = [threading.Thread(target=work, args=(i,)) for i in range(threads)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not wrong
        graphs.append(dbg.Graph(21, 100))
    for g in graphs:
        g.close()
