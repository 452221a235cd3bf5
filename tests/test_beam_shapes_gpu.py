"""Incoherent beam over the lanes per row (1 to 32), the blocks' shares of the channels and both
sides of the rules that choose between them, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05992_gb300 import corr

pytestmark = pytest.mark.gpu


# one and two lanes: rows of 64 bytes and less and longer ones, channels below, at and just past one
# and two blocks; 4 and 8 lanes; 16 lanes with few and many blocks; 32 lanes
@pytest.mark.parametrize("N,F,T,n_avg", [(16, 257, 6, 1), (48, 1, 4, 2), (48, 513, 3, 1), (80, 128, 4, 1), (112, 129, 6, 3),
                                         (240, 130, 20, 1), (1008, 257, 2, 2), (32, 129, 5, 1), (96, 65, 8, 2),
                                         (96, 64, 3, 1), (928, 150, 4, 4), (64, 70, 9, 3), (192, 65, 4, 1), (128, 33, 10, 5),
                                         (256, 33, 20, 10), (256, 500, 60, 1), (768, 17, 6, 2), (768, 961, 60, 2),
                                         (512, 9, 12, 3), (1024, 33, 10, 10)])
@pytest.mark.parametrize("zero_invalid", [False, True])
def test_beam_shapes(N, F, T, n_avg, zero_invalid):
    volt = np.random.default_rng(N + F + T).integers(0, 256, (T, F, N), dtype=np.uint8)
    got = corr.incoherent_beam(torch.from_numpy(volt).cuda(), n_avg, zero_invalid)
    assert np.array_equal(got.cpu().numpy(), oracle.beam(volt, n_avg, zero_invalid))
