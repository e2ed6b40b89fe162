"""Sketches whose CTAs exchange registers while they run: read sets of one
tile, of several tiles a CTA and of more tiles than CTAs, registers bit for bit
against the oracle."""

import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("n_reads", [256, 257, 40_000, 290_000])
def test_one_read_set(n_reads):
    rs = synth.ragged_reads(n_reads, 60, 17, n_reads)
    regs = dbg.sketch(17, *to_device(rs)).cpu().numpy().view(np.uint32)
    assert np.array_equal(regs[:1024], oracle.sketch(rs.packed, rs.offsets, 17))


def test_batch_of_uneven_read_sets():
    import torch
    sets = [synth.ragged_reads(n, 60, k, 5 * n + k) for n, k in
            [(3, 9), (100_000, 21), (0, 31), (700, 31), (250_000, 13), (256, 5)]]
    regs = torch.empty(len(sets), dbg.SKETCH_REGISTERS + 1, dtype=torch.int32, device="cuda")
    items = [(rs.k,) + to_device(rs) + (regs[i],) for i, rs in enumerate(sets)]
    for _ in range(2):
        dbg.sketch_batch(items)
    got = regs.cpu().numpy().view(np.uint32)
    for rs, r in zip(sets, got):
        assert np.array_equal(r[:1024], oracle.sketch(rs.packed, rs.offsets, rs.k)) and r[1024] == 0
