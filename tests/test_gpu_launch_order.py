"""Kernels whose launch overlaps the previous one keep the stream's order: inputs
written just before a call and overwritten just after it, calls back to back on
one graph, and the same calls captured into a CUDA graph."""

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


def outputs(rows, k):
    import torch
    keys = torch.zeros((rows, 2) if k > 32 else (rows,), dtype=torch.int64, device="cuda")
    return keys, torch.zeros((rows, 4), dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("path", [1, 2])
@pytest.mark.parametrize("k,n", [(21, 3), (21, 3000), (31, 60_000), (51, 20_000)])
def test_inputs_live_only_as_long_as_the_call(k, n, path, captured):
    import torch
    sets = [synth.sample_reads(synth.random_genome(20_000, i), n, 120, 0.0, i, k, "o")
            for i in range(3)]
    devs = [to_device(rs) for rs in sets]
    slots = 100_000
    refs = []
    for dev in devs:
        g = dbg.Graph(k, slots)
        g.set_tuning(insert_path=1)
        g.build(*dev)
        refs.append(g.export())
        g.close()
    g = dbg.Graph(k, slots)
    g.set_tuning(insert_path=path)
    packed, offsets = (torch.zeros_like(t) for t in devs[0])
    s = torch.cuda.Stream()
    torch.cuda.synchronize()

    def call(i):  # the reads twice: a rebuild, then an insert into it
        packed.copy_(devs[i][0])
        offsets.copy_(devs[i][1])
        g.build(packed, offsets, stream=s)
        g.insert(packed, offsets, stream=s)
        packed.zero_()
        offsets.zero_()

    with torch.cuda.stream(s):
        call(0)  # (a first call makes the path's buffers, which a capture cannot)
        for i in list(range(3)) * 3:
            if captured:
                cg = torch.cuda.CUDAGraph()
                with torch.cuda.graph(cg, stream=s):
                    call(i)
                cg.replay()
            else:
                call(i)
            keys, counts = outputs(len(refs[i][0]), k)
            D = g.export_into(keys, counts, stream=s)
            assert D == len(refs[i][0])
            assert np.array_equal(keys.cpu().numpy().view(np.uint64), refs[i][0])
            assert np.array_equal(counts.cpu().numpy().view(np.uint32), 2 * refs[i][1])
    g.close()
