"""Fine filterbank: inputs so long that a CTA takes several groups of frames give the
codes of their pieces, which take one group per CTA; and the codes and spectra of
whole and ragged sets of inputs are those of the inputs taken alone."""
import pytest
import torch

from paper_1501_05992_gb300 import corr
from synth import coarse

pytestmark = pytest.mark.gpu


def _codes(x, h):
    return corr.fine_pfb(x, h, 0.01)[0]


@pytest.mark.parametrize("taps", [1, 12])
@pytest.mark.parametrize("n", [2, 16])
def test_several_groups_per_cta(taps, n):
    frames = 8 * 65535 + 13
    g = torch.Generator(device="cuda").manual_seed(taps + n)
    x = torch.randint(-90, 91, (1, n, 128 * (frames + taps - 1), 2), dtype=torch.int8, device="cuda", generator=g)
    h = torch.rand(128 * taps, device="cuda", generator=g)
    whole = _codes(x, h)
    cut = 262141
    first = _codes(x[:, :, :128 * (cut + taps - 1)].contiguous(), h)
    rest = _codes(x[:, :, 128 * cut:].contiguous(), h)
    assert torch.equal(whole[:cut], first)
    assert torch.equal(whole[cut:], rest)


@pytest.mark.parametrize("n", [3, 16, 31, 48])
def test_inputs_by_themselves(n):
    h = torch.from_numpy(coarse.kaiser_sinc_window(12)).float().cuda()
    x = torch.from_numpy(coarse.coarse_samples(n, 2, n, 128 * (20 + 11))).cuda()
    got = _codes(x, h)
    for i in {0, 1, n // 2, n - 1}:
        assert torch.equal(got[:, :, i], _codes(x[:, i:i + 1].contiguous(), h)[:, :, 0])


@pytest.mark.parametrize("volt", [False, True])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 15, 16, 18, 33])
@pytest.mark.parametrize("taps,frames", [(12, 3), (12, 20), (1, 17)])
def test_spectra_by_themselves(n, taps, frames, volt):
    h = torch.from_numpy(coarse.kaiser_sinc_window(12)[:128 * taps]).float().cuda()
    x = torch.from_numpy(coarse.coarse_samples(n, 2, n, 128 * (frames + taps - 1))).cuda()
    codes, spec = corr.fine_pfb(x, h, 0.01, volt=volt, spec=True)
    for i in {0, 1, n // 2, n - 1}:
        one_codes, one_spec = corr.fine_pfb(x[:, i:i + 1].contiguous(), h, 0.01, volt=volt, spec=True)
        assert torch.equal(spec[:, :, i], one_spec[:, :, 0])
        if volt:
            assert torch.equal(codes[:, :, i], one_codes[:, :, 0])
