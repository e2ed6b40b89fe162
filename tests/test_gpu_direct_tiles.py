"""The direct insert cuts its reads into tiles by their number: read sets at
the edges of that rule, element by element against the oracle."""

import pytest

from gpu_util import assert_same_graph, gpu_export, oracle_export
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


# one read; one tile and its rest; more tiles than CTAs at two reads a tile;
# one wave of the largest tiles, and one read more (two waves)
@pytest.mark.parametrize("n", [1, 2, 3, 2433, 24320, 24321])
@pytest.mark.parametrize("block", [0, 512])
def test_read_counts(n, block):
    rs = synth.ragged_reads(n, 60, 11, 70 + n, lead=n % 5)
    got = gpu_export(rs, capacity=max(64, min(2 << 20, 120 * n)),
                     tuning=dict(insert_path=1, block_threads=block, warp_aggregate=0))
    assert_same_graph(got, oracle_export(rs))
