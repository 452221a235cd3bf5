"""The small-array CUDA-core X-engine (up to 64 inputs): tile and group edges,
time slices over one to eight CTAs, byte-aligned rows, storing and adding,
bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05992_gb300 import corr

pytestmark = pytest.mark.gpu


# inputs around the 4 x 4 tiles' edges and the range's ends; samples around one
# sample, an odd count, the shortest slices (64 samples) and several pieces;
# channels below and above what one cluster per channel needs
@pytest.mark.parametrize("N,F,T", [(1, 1, 1), (1, 3, 127), (3, 2, 128), (4, 1, 129), (5, 310, 40), (7, 40, 255),
                                   (16, 160, 256), (17, 2, 1025), (31, 1, 511), (33, 5, 64), (48, 77, 130),
                                   (61, 2, 900), (63, 1, 1024), (64, 4, 513)])
@pytest.mark.parametrize("offset", [0, 1, 4])
def test_small_arrays_exact(N, F, T, offset):
    zi = offset == 1
    volt = np.random.default_rng(N * F + T + offset).integers(0, 256, (T, F, N), dtype=np.uint8)
    buf = torch.zeros(T * F * N + 8, dtype=torch.uint8, device="cuda")
    d = buf[offset:offset + T * F * N].view(T, F, N)
    d.copy_(torch.from_numpy(volt))
    c = corr.Correlator(N, F, 2 * T, path="cudacore", zero_invalid=zi)
    whole = c.integrate(d)
    c.accumulate(d)
    c.accumulate(d[T // 2:])
    acc = c.dump()
    c.sync()
    c.close()
    vis = oracle.xmac(volt, zi)
    assert np.array_equal(whole.cpu().numpy(), oracle.to_int32(vis))
    assert np.array_equal(acc.cpu().numpy(), oracle.to_int32(vis + oracle.xmac(volt[T // 2:], zi)))
