"""Tensor-core X-engine on rows of one to three bytes, whose words hold several channels, on every
byte offset of the buffer and with channels next to the first and the last one: bit-exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05992_gb300 import corr

from _gpu import path_available

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,F,T", [(1, 4, 3), (1, 9, 65), (2, 4, 64), (2, 7, 130), (3, 5, 66)])
@pytest.mark.parametrize("offset", [0, 1, 2, 3])
def test_rows_shorter_than_a_word(N, F, T, offset):
    if not path_available("tc_fp8", N):
        pytest.skip("tc_fp8 unsupported")
    volt = np.random.default_rng(100 * N + F + offset).integers(0, 256, (T, F, N), dtype=np.uint8)
    buf = torch.full((T * F * N + 8,), 0x5A, dtype=torch.uint8, device="cuda")
    d = buf[offset:offset + T * F * N].view(T, F, N)
    d.copy_(torch.from_numpy(volt))
    c = corr.Correlator(N, F, T, path="tc_fp8")
    tri, beam = c.integrate_beam(d, 1)
    c.sync()
    c.close()
    assert np.array_equal(tri.cpu().numpy(), oracle.to_int32(oracle.xmac(volt)))
    assert np.array_equal(beam.cpu().numpy(), oracle.beam(volt, 1))
