"""Arrays of more than 256 inputs in one call.  The last of an odd number of tiles, alone or as
a block with an empty second tile: channel counts on both sides of the rule that chooses, one
input to a whole tile in it; long integrations whose last round of items goes in slices of
samples.  Stored, added and with the fused beam, bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05992_gb300 import corr

from _gpu import path_available

pytestmark = pytest.mark.gpu


# on 76 pairs of CTAs: one round of pairs, two rounds, a round more with the last tile, three rounds
@pytest.mark.parametrize("N,F,T", [(257, 25, 70), (272, 45, 65), (384, 50, 64), (640, 21, 130), (897, 5, 63),
                                   (257, 26, 70), (304, 51, 65), (384, 38, 64), (513, 11, 130), (640, 28, 63)])
@pytest.mark.parametrize("zero_invalid", [False, True])
def test_last_tile_exact(N, F, T, zero_invalid):
    _check(N, F, T, zero_invalid)


# one to four rounds of both kinds of items in one launch, one to three rounds with the last tiles
# apart (short and longer integrations), and five rounds in launches of their own
@pytest.mark.parametrize("N,F,T", [(512, 38, 70), (768, 20, 65), (1024, 14, 64), (400, 60, 63), (1024, 1, 200),
                                   (640, 32, 130), (640, 12, 65), (500, 45, 64), (512, 95, 65), (384, 76, 65),
                                   (384, 60, 705), (272, 98, 64), (380, 98, 63)])
@pytest.mark.parametrize("zero_invalid", [False, True])
def test_both_kinds_of_items_in_one_launch(N, F, T, zero_invalid):
    _check(N, F, T, zero_invalid)


# few items of the tiles off the blocks left for the last round, with last tiles and without; last
# tiles alone left for it; a last slice that ends within a stage; padded rows; two whole rounds
@pytest.mark.parametrize("N,F,T,zero_invalid", [(512, 20, 5000, False), (400, 20, 4999, True), (512, 39, 4100, True),
                                                (640, 13, 5057, False), (272, 38, 4300, True), (300, 37, 4097, False),
                                                (257, 76, 6020, False), (768, 9, 4160, True), (1024, 5, 4200, False),
                                                (520, 13, 4100, False)])
def test_last_round_in_slices(N, F, T, zero_invalid):
    _check(N, F, T, zero_invalid)


# (inputs, channels, samples) beside arrays of up to 128 inputs: one to four rounds of both kinds of
# items, with last tiles and without, longer or shorter than the others' integrations; long ones that
# leave pairs idle, and an array of 129..256 inputs beside, which keep their launches
@pytest.mark.parametrize("arrays", [[(512, 27, 168), (128, 27, 168)], [(100, 30, 200), (320, 66, 130)],
                                    [(384, 20, 65), (64, 200, 64), (128, 7, 300)], [(1024, 14, 64), (17, 5, 63)],
                                    [(500, 21, 1025), (96, 40, 65)], [(512, 30, 1100), (128, 90, 64)],
                                    [(128, 40, 130), (512, 38, 70), (256, 30, 100)], [(257, 9, 64), (384, 9, 130)]])
@pytest.mark.parametrize("zero_invalid", [False, True])
def test_large_array_beside_others(arrays, zero_invalid):
    if not all(path_available("tc_fp8", n) for n, _, _ in arrays):
        pytest.skip("tc_fp8 unsupported")
    rng = np.random.default_rng(len(arrays) + arrays[0][1])
    volts = [rng.integers(0, 256, (t, f, n), dtype=np.uint8) for n, f, t in arrays]
    d = [torch.from_numpy(v).cuda() for v in volts]
    b = corr.Batch([dict(n_inputs=n, n_chan=f, n_time_per_int=2 * t, path="tc_fp8", zero_invalid=zero_invalid)
                    for n, f, t in arrays])
    whole = b.integrate(d)
    b.accumulate(d)
    b.accumulate(d)
    added = b.dump()
    b.sync()
    b.close()
    for v, w, a in zip(volts, whole, added):
        vis = oracle.xmac(v, zero_invalid)
        assert np.array_equal(w.cpu().numpy(), oracle.to_int32(vis))
        assert np.array_equal(a.cpu().numpy(), oracle.to_int32(2 * vis))


def _check(N, F, T, zero_invalid):
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


def test_slices_under_capture():
    """The launches of a call in slices, which overlap and wait for the zeroing, replayed from a
    graph on new samples and twice in a row."""
    N, F, T = 640, 13, 4200
    if not path_available("tc_fp8", N):
        pytest.skip("tc_fp8 unsupported")
    b = corr.Batch([dict(n_inputs=N, n_chan=F, n_time_per_int=T, path="tc_fp8")])
    rng = np.random.default_rng(5)
    volt = rng.integers(0, 256, (T, F, N), dtype=np.uint8)
    d = torch.from_numpy(volt).cuda()
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    graph, outs = b.capture([d], stream=stream)
    for _ in range(2):
        d.copy_(torch.from_numpy(volt))
        torch.cuda.synchronize()
        graph.launch(stream)
        graph.launch(stream)
        stream.synchronize()
        assert np.array_equal(outs[0].cpu().numpy(), oracle.to_int32(oracle.xmac(volt)))
        volt = rng.integers(0, 256, (T, F, N), dtype=np.uint8)
    b.sync(stream)
    graph.close()
