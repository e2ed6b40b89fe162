"""Exports into host outputs of which all, a part or only the two ends are pinned:
the sort writes outputs itself only when they lie in one pinned range.  Other
outputs are copied to, which CUDA may refuse for partly pinned memory (where a
write by the device may fault)."""

import ctypes

import numpy as np
import pytest

import oracle
from gpu_util import to_device
from paper_2401_02756_gb300 import build, dbg, synth

pytestmark = pytest.mark.gpu

PAGE = 65536


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    build.build()
    dbg.load()


def aligned(nbytes):
    raw = np.zeros(nbytes + PAGE, dtype=np.uint8)
    return raw[-raw.ctypes.data % PAGE:][:nbytes]


# parts of the outputs' pages that are registered
@pytest.mark.parametrize("parts", [[(0, 1)], [(0, 0.25), (0.75, 1)], [(0, 0.25)], [(0.75, 1)],
                                   [(0, 0.5), (0.5, 1)], []])
@pytest.mark.parametrize("k", [31, 51])
def test_registered_parts(parts, k):
    import torch
    rt = torch.cuda.cudart()
    rs = synth.ragged_reads(2000, 150, k, 6)
    ref = oracle.build_graph(rs.packed, rs.offsets, k)
    D = len(ref.keys)
    g = dbg.Graph(k, 2 * D)
    g.insert(*to_device(rs))
    pages = -(-16 * D // PAGE)
    pages += -pages % 4
    bufs, registered = [], []
    for _ in range(2):
        buf = aligned(pages * PAGE)
        bufs.append(buf)
        for a, b in parts:
            at, n = int(a * pages) * PAGE, int((b - a) * pages) * PAGE
            assert int(rt.cudaHostRegister(buf.ctypes.data + at, n, 0)) == 0
            registered.append(buf.ctypes.data + at)
    rows = pages * PAGE // 16  # (the last row ends with the last page)
    n = ctypes.c_uint64()
    st = dbg.load().dbg_export_sorted(g.handle, bufs[0].ctypes.data, bufs[1].ctypes.data, rows,
                                      ctypes.byref(n), None)
    for at in registered:
        assert int(rt.cudaHostUnregister(at)) == 0
    if st == dbg.ERR_CUDA and parts not in ([], [(0, 1)]):  # (a copy that CUDA refuses)
        dbg.load().dbg_reset(g.handle, None)  # (takes the error that CUDA still reports)
        g.close()
        return
    assert st == dbg.OK and n.value == D
    keys = bufs[0].view(np.uint64)
    keys = keys[:2 * D].reshape(D, 2) if k > 32 else keys[:D]
    assert np.array_equal(keys, ref.keys)
    assert np.array_equal(bufs[1].view(np.uint32)[:4 * D].reshape(D, 4), ref.counts)
    g.close()


@pytest.mark.parametrize("lead", [0, 16, 4096])
def test_a_slice_of_a_pinned_buffer(lead):
    import torch
    rs = synth.ragged_reads(2000, 150, 31, 6)
    ref = oracle.build_graph(rs.packed, rs.offsets, 31)
    D = len(ref.keys)
    g = dbg.Graph(31, 2 * D)
    g.insert(*to_device(rs))
    buf = torch.zeros(lead + 48 * D, dtype=torch.uint8, pin_memory=True).numpy()[lead:]
    keys = buf[:8 * D].view(np.uint64)
    at = -(-8 * D // 16) * 16
    counts = buf[at:at + 16 * D].view(np.uint32).reshape(D, 4)
    got = g.export(out=(keys, counts))
    assert np.array_equal(got[0], ref.keys) and np.array_equal(got[1], ref.counts)
    assert not buf[at + 16 * D:].any()
    g.close()
