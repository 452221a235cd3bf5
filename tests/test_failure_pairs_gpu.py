"""Failure detection in the kernels over pairs of CTAs, without a GPU fault: their bounded waits
are made to expire while loads, MMAs and rows between the CTAs of a pair are in flight; every
launch of the call ends with CORR_E_TIMEOUT and the context goes on."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05992_gb300 import corr

from _gpu import path_available

pytestmark = pytest.mark.gpu


# 256-input blocks; the same in slices of samples that add; with the tiles off the blocks, and
# with a last tile alone; more items than CTA pairs
@pytest.mark.parametrize("N,F,T", [(256, 8, 256), (256, 4, 4096), (200, 100, 130), (384, 5, 300), (512, 80, 200),
                                   (640, 3, 64)])
def test_stall_times_out_and_context_recovers(N, F, T):
    if not path_available("tc_fp8", N):
        pytest.skip("tc_fp8 unsupported")
    volt = np.random.default_rng(N + F).integers(0, 256, (T, F, N), dtype=np.uint8)
    v = torch.from_numpy(volt).cuda()
    c = corr.Correlator(N, F, T, path="tc_fp8")
    for _ in range(2):
        c.set_wait_limit(20_000_000)              # about 10 ms of SM clock
        c.inject_stall()
        c.integrate(v)
        with pytest.raises(corr.CorrError) as e:
            c.sync()
        assert e.value.status == corr.CORR_E_TIMEOUT
        c.set_wait_limit(0)
        got = c.integrate(v)
        c.sync()
        assert np.array_equal(got.cpu().numpy(), oracle.to_int32(oracle.xmac(volt)))
    c.close()
