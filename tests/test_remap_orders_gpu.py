"""Output remap in Appendix A's order (arithmetic) and the same order given as a
table, against the oracle: one PFB and several, sums whose (dump, channel)
triples fill the groups of four loads exactly, in part and not at all, and more
channel groups than a launch has rows of blocks."""
import numpy as np
import pytest
import torch

import oracle
from paper_1501_05992_gb300 import corr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,f", [(64, 6), (192, 12), (320, 6)])
@pytest.mark.parametrize("f_avg,n_dumps", [(1, 1), (2, 1), (2, 2), (3, 1), (1, 5), (6, 8)])
@pytest.mark.parametrize("table", [False, True])
def test_pfb_order(n, f, f_avg, n_dumps, table):
    rng = np.random.default_rng(n + 10 * f_avg + n_dumps)
    tris = rng.integers(-1 << 24, 1 << 24, (n_dumps, f, n * (n + 1) // 2, 2)).astype(np.int32)
    order = torch.from_numpy(oracle.pfb_order(n)).cuda() if table else None
    got = corr.remap([torch.from_numpy(t).cuda() for t in tris], order, f_avg=f_avg).cpu().numpy()
    want = oracle.remap(tris, oracle.pfb_order(n), f_avg=f_avg)
    assert np.array_equal(got, oracle.to_int32(want))


@pytest.mark.parametrize("f_avg", [1, 3])
def test_more_groups_than_block_rows(f_avg):
    n, f = 64, 12801
    tri = torch.randint(-1000, 1000, (f, n * (n + 1) // 2, 2), dtype=torch.int32, device="cuda")
    got = corr.remap(tri, f_avg=f_avg).cpu().numpy()
    want = oracle.remap(tri.cpu().numpy(), oracle.pfb_order(n), f_avg=f_avg)
    assert np.array_equal(got, oracle.to_int32(want))
