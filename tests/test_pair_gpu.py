"""The CTA-pair tensor-core X-engine (129 to 256 inputs): tile, stage and team
edges, ragged last tiles, adding launches and the fused beam, bit-exact against
the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05992_gb300 import corr

from _gpu import path_available

pytestmark = pytest.mark.gpu


# inputs around the two tiles' edges (one input, half a tile and all but one in
# the second); samples around a 64-sample stage and the four teams' turns; more
# channels than CTA pairs where a pair must take several items
@pytest.mark.parametrize("N,F,T", [(129, 2, 65), (144, 3, 64), (176, 1, 1), (192, 2, 63), (193, 90, 130), (208, 3, 257),
                                   (250, 2, 320), (255, 1, 191), (256, 160, 300), (256, 1, 4100)])
@pytest.mark.parametrize("zero_invalid", [False, True])
def test_pair_blocks_exact(N, F, T, zero_invalid):
    if not path_available("tc_fp8", N):
        pytest.skip("tc_fp8 unsupported")
    volt = np.random.default_rng(N + F + T).integers(0, 256, (T, F, N), dtype=np.uint8)
    c = corr.Correlator(N, F, 2 * T, path="tc_fp8", zero_invalid=zero_invalid)
    d = torch.from_numpy(volt).cuda()
    tri, beam = c.integrate_beam(d, 1)
    whole = c.integrate(d)
    h = T // 3
    if h:
        c.accumulate(d[:h])
    c.accumulate(d[h:])
    c.accumulate(d)
    acc = c.dump()
    c.sync()
    c.close()
    vis = oracle.xmac(volt, zero_invalid)
    assert np.array_equal(whole.cpu().numpy(), oracle.to_int32(vis))
    assert np.array_equal(tri.cpu().numpy(), oracle.to_int32(vis))
    assert np.array_equal(acc.cpu().numpy(), oracle.to_int32(2 * vis))
    assert np.array_equal(beam.cpu().numpy(), oracle.beam(volt, 1, zero_invalid))


@pytest.mark.parametrize("byte", [0x77, 0x88, 0x80, 0x08, 0x87, 0x78])
def test_pair_extreme_sums_exact(byte):
    """Constant samples of the largest codes over 33000 samples: the largest FP32
    partial sums a launch of 32768 samples can reach, and its split."""
    if not path_available("tc_fp8", 256):
        pytest.skip("tc_fp8 unsupported")
    N, F, T = 256, 1, 33000
    volt = np.full((T, F, N), byte, np.uint8)
    volt[:, :, 128:] = (byte >> 4) | ((byte << 4) & 0xFF)
    c = corr.Correlator(N, F, T, path="tc_fp8")
    got = c.integrate(torch.from_numpy(volt).cuda())
    c.sync()
    c.close()
    # every sample is the same: T times the product of one
    want = oracle.xmac(volt[:1]) * T
    assert np.array_equal(got.cpu().numpy(), oracle.to_int32(want))


# rows on every byte offset (odd and even strides, buffers that start off a word
# boundary, the first and last channels' words over the ends of the buffer), the
# second tile ending at, before and after a word of its last lane
@pytest.mark.parametrize("N,F,T", [(131, 1, 70), (159, 4, 129), (201, 3, 64), (250, 6, 333), (251, 2, 65),
                                   (253, 80, 40), (254, 5, 257), (255, 3, 200)])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_pair_rows_on_any_byte(N, F, T, offset):
    if not path_available("tc_fp8", N):
        pytest.skip("tc_fp8 unsupported")
    volt = np.random.default_rng(N + F + T + offset).integers(0, 256, (T, F, N), dtype=np.uint8)
    buf = torch.full((T * F * N + 8,), 0x5A, dtype=torch.uint8, device="cuda")
    d = buf[offset:offset + T * F * N].view(T, F, N)
    d.copy_(torch.from_numpy(volt))
    c = corr.Correlator(N, F, T, path="tc_fp8", zero_invalid=offset == 3)
    tri, beam = c.integrate_beam(d, 1)
    c.accumulate(d)
    acc = c.dump()
    c.sync()
    c.close()
    want = oracle.to_int32(oracle.xmac(volt, offset == 3))
    assert np.array_equal(tri.cpu().numpy(), want)
    assert np.array_equal(acc.cpu().numpy(), want)
    assert np.array_equal(beam.cpu().numpy(), oracle.beam(volt, 1, offset == 3))


# tiles off the 256-input blocks and a last tile alone: one input past a block, an
# odd number of tiles, a ragged last tile in and off a block; the input counts that
# are no multiple of 16 run on padded rows; T around a stage and the teams' turns
@pytest.mark.parametrize("N,F,T", [(257, 2, 63), (272, 1, 65), (384, 3, 128), (400, 2, 129), (512, 80, 100),
                                   (513, 1, 200), (640, 2, 64), (700, 1, 1), (1024, 1, 321)])
def test_tiles_off_the_blocks_exact(N, F, T):
    _check_all_calls(N, F, T, zero_invalid=N % 3 == 0)


# a single tile: its inputs' last 16 columns, rows on any byte, channels past the SMs
@pytest.mark.parametrize("N,F,T", [(1, 2, 70), (15, 3, 65), (16, 1, 64), (49, 2, 300), (64, 160, 129), (97, 1, 63),
                                   (113, 2, 257), (127, 5, 130), (128, 310, 65)])
def test_single_tiles_exact(N, F, T):
    _check_all_calls(N, F, T, zero_invalid=N % 2 == 0)


def _check_all_calls(N, F, T, zero_invalid):
    if not path_available("tc_fp8", N):
        pytest.skip("tc_fp8 unsupported")
    volt = np.random.default_rng(N + F + T).integers(0, 256, (T, F, N), dtype=np.uint8)
    c = corr.Correlator(N, F, 2 * T, path="tc_fp8", zero_invalid=zero_invalid)
    d = torch.from_numpy(volt).cuda()
    tri, beam = c.integrate_beam(d, 1)
    c.accumulate(d)
    c.accumulate(d)
    acc = c.dump()
    c.sync()
    c.close()
    vis = oracle.xmac(volt, zero_invalid)
    assert np.array_equal(tri.cpu().numpy(), oracle.to_int32(vis))
    assert np.array_equal(acc.cpu().numpy(), oracle.to_int32(2 * vis))
    assert np.array_equal(beam.cpu().numpy(), oracle.beam(volt, 1, zero_invalid))


# long integrations whose last round of channels is split into slices of samples: fewer
# channels than CTA pairs, a few more, on and off 16-byte rows, a last slice of one sample
@pytest.mark.parametrize("N,F,T", [(256, 1, 2048), (256, 3, 4097), (250, 5, 3073), (131, 38, 2111), (255, 77, 1999),
                                   (256, 79, 5000), (250, 80, 4990), (192, 155, 1057), (128, 3, 4097), (100, 155, 2111),
                                   (65, 160, 1999)])
@pytest.mark.parametrize("zero_invalid", [False, True])
def test_last_round_in_slices(N, F, T, zero_invalid):
    _check_all_calls(N, F, T, zero_invalid)


def test_overlapping_launches_under_capture():
    """A batch whose arrays take the pair, off-block and single-tile launches, which overlap
    (two kinds of each: with invalid samples zeroed and not), replayed from a graph."""
    shapes = [(384, 40, 300, False), (128, 200, 100, True), (250, 30, 257, False), (640, 12, 128, True)]
    if not path_available("tc_fp8", 640):
        pytest.skip("tc_fp8 unsupported")
    rng = np.random.default_rng(17)
    make = lambda: [rng.integers(0, 256, (t, f, n), dtype=np.uint8) for n, f, t, _ in shapes]
    b = corr.Batch([dict(n_inputs=n, n_chan=f, n_time_per_int=t, path="tc_fp8", zero_invalid=z)
                    for n, f, t, z in shapes])
    volts = make()
    dev = [torch.from_numpy(v).cuda() for v in volts]
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    graph, outs = b.capture(dev, stream=stream)
    for _ in range(3):
        for d, v in zip(dev, volts):
            d.copy_(torch.from_numpy(v))
        torch.cuda.synchronize()
        graph.launch(stream)
        graph.launch(stream)
        stream.synchronize()
        for (n, f, t, z), v, o in zip(shapes, volts, outs):
            assert np.array_equal(o.cpu().numpy(), oracle.to_int32(oracle.xmac(v, z))), n
        volts = make()
    b.sync(stream)
    graph.close()
