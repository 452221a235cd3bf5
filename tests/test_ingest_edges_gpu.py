"""Packet ingest at the edges of its groups of packets: streams that end within
a warp's group, a block's stretch or a 16-byte piece, on each alignment a stream
may have, and banks with few packets or none, whose missing slots are written by
the last pass."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05992_gb300 import corr
from synth import packets as pkts

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lane():
    block = np.random.default_rng(11).integers(0, 256, (500, 3072, 256), dtype=np.uint8)
    return np.concatenate([pkts.lane_packets(block, p, 5, 9) for p in range(4)])


@pytest.mark.parametrize("offset", [0, 4, 8, 12])
@pytest.mark.parametrize("count", [0, 1, 3, 4, 5, 31, 33, 63, 64, 65, 2001])
def test_stream_ends(lane, offset, count):
    sel = lane[np.random.default_rng(count).choice(len(lane), count, replace=False)]
    # bytes past the stream are another packet's: none of them may be taken for the last one's
    raw = torch.full((sel.size + offset + 264,), 0x5A, dtype=torch.uint8, device="cuda")
    raw[offset:offset + sel.size] = torch.from_numpy(np.ascontiguousarray(sel).reshape(-1)).cuda()
    p = raw[offset:offset + sel.size].view(-1, 264)
    out = torch.full((500, 3072, 256), 0x33, dtype=torch.uint8, device="cuda")
    seen = torch.full((corr.PKT_SLOTS,), 7, dtype=torch.uint8, device="cuda")
    volt, cnt = corr.ingest_packets(p, 9, out=out, seen=seen)
    torch.cuda.synchronize()
    want_v, want_c = oracle.ingest(sel, 9)
    assert np.array_equal(cnt.cpu().numpy().astype(np.int64), want_c)
    assert np.array_equal(volt.cpu().numpy(), want_v)


def test_capture(lane):
    """The call's three launches, which overlap, replayed from a graph on new packets."""
    sel = lane[:4003]
    p = torch.from_numpy(np.ascontiguousarray(sel)).cuda()
    out = torch.empty((500, 3072, 256), dtype=torch.uint8, device="cuda")
    seen = torch.empty((corr.PKT_SLOTS,), dtype=torch.uint8, device="cuda")
    cnt = torch.empty((corr.PKT_COUNTERS,), dtype=torch.int32, device="cuda")
    corr.ingest_packets(p, 9, out=out, seen=seen, counters=cnt)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        corr.ingest_packets(p, 9, out=out, seen=seen, counters=cnt, stream=torch.cuda.current_stream())
    for first in (0, 5000, 60000):
        sel = lane[first:first + 4003]
        p.copy_(torch.from_numpy(np.ascontiguousarray(sel)))
        g.replay()
        torch.cuda.synchronize()
        want_v, want_c = oracle.ingest(sel, 9)
        assert np.array_equal(cnt.cpu().numpy().astype(np.int64), want_c)
        assert np.array_equal(out.cpu().numpy(), want_v)
