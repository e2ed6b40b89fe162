"""Rebuilds from long reads take no longer than emptying the table and inserting:
the insert's few or long-lived CTAs are spread over the SMs, whatever kernel
they are launched behind."""

import time

import pytest

from paper_2401_02756_gb300 import build, dbg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


def sampled(genome, n, length, seed, err=0.0):
    """(packed, offsets) of n reads of a genome, made on the GPU."""
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    text = torch.randint(0, 4, (genome,), dtype=torch.uint8, device="cuda", generator=gen)
    starts = torch.randint(0, genome - length + 1, (n, 1), device="cuda", generator=gen)
    reads = text[starts + torch.arange(length, device="cuda")].view(-1)
    if err:
        wrong = torch.rand(reads.numel(), device="cuda", generator=gen) < err
        reads = (reads + wrong.to(torch.uint8)) & 3
    reads = reads.view(-1, 4)
    packed = reads[:, 0] | (reads[:, 1] << 2) | (reads[:, 2] << 4) | (reads[:, 3] << 6)
    return packed, torch.arange(n + 1, device="cuda") * length


def seconds(f, before=lambda: None):
    import torch
    t = []
    for _ in range(7):
        before()
        torch.cuda.synchronize()
        a = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - a)
    return sorted(t)[3]


@pytest.mark.parametrize("k", [21, 31, 51])
def test_few_long_reads(k):
    dev = sampled(500_000, 402, 10_000, k)
    g = dbg.Graph(k, 2_500_000)
    g.set_tuning(insert_path=1)
    insert = seconds(lambda: g.insert(*dev), g.reset)
    want = g.stats()
    rebuild = seconds(lambda: g.build(*dev))
    assert g.stats() == want
    assert rebuild < 1.2 * insert + 20e-6, (rebuild, insert)
    g.close()


def test_a_rebuild_of_more_events_than_its_scratch_holds():
    # given to the direct insert after the binned chain's kernels
    dev = sampled(2_000_000, 65_000, 5000, 9, err=0.0001)
    g = dbg.Graph(31, 4_000_000)
    g.reserve_events(17_000_000)
    rebuild = seconds(lambda: g.build(*dev))
    got = g.stats()
    g.set_tuning(insert_path=1, warp_aggregate=0)
    direct = seconds(lambda: g.build(*dev))
    assert g.stats() == got
    assert rebuild < 1.2 * direct, (rebuild, direct)
    g.close()
