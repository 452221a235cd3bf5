"""Workspace figures without a device: what a shape's calls never touch is not asked for."""
import pytest

from paper_1501_05992_gb300 import corr

CAP = 4 << 30


def _others(n, f, t):
    """Status word, accumulators, operand staging and host buffers of a shape, from the header's
    description, each on 256 bytes."""
    up = lambda x, a: -(-x // a) * a

    def staging(unit):
        pad = up(n, 64)
        chunk = min(up(t, 64), 8192)
        while chunk > 64 and 4 * chunk * pad > 1 << 30:
            chunk -= 64
        return 4 * chunk * pad * min(f, max(1, (1 << 30) // (4 * chunk * pad)), 65535)

    return (256 + up(f * n * (n + 1) * 4, 256) + up(staging(64), 256) + 3 * up(min(t, 500) * f * n, 256))


@pytest.mark.parametrize("n,f,t", [(250, 768, 4990), (129, 3, 100), (100, 300, 5000), (1, 2, 70), (255, 3072, 20000)])
def test_arrays_read_as_they_are_reserve_no_padded_rows(n, f, t):
    assert corr.workspace_bytes(n, f, t) == _others(n, f, t)


@pytest.mark.parametrize("n,f,t", [(256, 768, 5000), (512, 20, 300)])
def test_whole_rows_need_no_copy(n, f, t):
    assert corr.workspace_bytes(n, f, t) == _others(n, f, t)


@pytest.mark.parametrize("n,f,t", [(257, 10, 100), (700, 100, 4000)])
def test_longer_rows_keep_theirs(n, f, t):
    """The padded copy of longer rows stays: a whole integration, in rows of 16 bytes' multiples."""
    pad = -(-n // 16) * 16 * f * (-(-t // 64) * 64)
    assert pad <= CAP and corr.workspace_bytes(n, f, t) == _others(n, f, t) + -(-pad // 256) * 256
