"""The autotuner's candidates and cache keys, without a GPU."""
import torch

from paper_1501_05992_gb300 import autotune


def test_candidates_hold_every_kernel_once():
    """CUDA-core shape 0 is the only one that runs the kernel of small arrays; the tensor-core path
    chooses its items itself, so that its tile values measure the same kernels."""
    assert ("cudacore", 0) in autotune.CANDIDATES
    assert [tile for path, tile in autotune.CANDIDATES if path == "tc_fp8"] == [0]
    assert len(set(autotune.CANDIDATES)) == len(autotune.CANDIDATES)


def test_results_of_other_candidates_are_no_answer(monkeypatch):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda device: "card")
    key = autotune._key(torch.device("cuda", 0), 16, 32, 1000)
    assert key.startswith("card|16x32x1000") and key != "card|16x32x1000"
    staged = [("cudacore", 64), ("cudacore", 32)]
    assert autotune._key(torch.device("cuda", 0), 16, 32, 1000, staged) != key
    assert autotune._key(torch.device("cuda", 0), 16, 32, 1000, list(autotune.CANDIDATES)) == key
