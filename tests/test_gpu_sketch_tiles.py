"""Sketches of one read set at the sizes where its reads are cut into tiles another
way, against the batched sketch (whose tiles are fixed) and the oracle."""

import numpy as np
import pytest

import oracle
from gpu_util import to_device
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu

CTAS = 152 * 7 // 4  # tiles that few reads are cut into


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


@pytest.mark.parametrize("n,length", [(1, 30), (7, 90), (9, 20_000), (500, 10_000), (8 * CTAS - 1, 40),
                                      (8 * CTAS + 1, 40), (100 * CTAS + 3, 36), (256 * CTAS, 30),
                                      (256 * CTAS + 1, 30)])
def test_single_equals_batched(n, length):
    import torch
    rs = synth.sample_reads(synth.random_genome(60_000, n), n, length, 0.001, n, 21, "s")
    packed, offsets = to_device(rs)
    one = dbg.sketch(21, packed, offsets)
    regs = torch.zeros(dbg.SKETCH_REGISTERS + 1, dtype=torch.int32, device="cuda")
    dbg.sketch_batch([(21, packed, offsets, regs)])
    assert torch.equal(one, regs)
    if n * length < 6_000_000:
        assert np.array_equal(one.cpu().numpy().view(np.uint32)[:-1],
                              oracle.sketch(rs.packed, rs.offsets, 21))
