"""A tuned small array runs the kernel of small arrays where it is the fastest measured."""
import json

import pytest
import torch

from paper_1501_05992_gb300 import autotune, corr

pytestmark = pytest.mark.gpu


def test_small_array_is_planned_on_its_kernel(tmp_path):
    cache = tmp_path / "tune.json"
    # a result of an earlier candidate set, as such a cache may hold it
    cache.write_text(json.dumps({f"{torch.cuda.get_device_name(0)}|16x32x1000":
                                 {"path": "cudacore", "tile": 32, "ms": {"cudacore/32": 1.0}, "probe_channels": 32}}))
    plan = autotune.plan([(16, 32, 1000)], cache_path=str(cache))
    assert (plan[0]["path"], plan[0]["tile"]) == ("cudacore", 0)
    b = corr.Batch(plan)
    b.profile_read()
    b.integrate([torch.zeros((1000, 32, 16), dtype=torch.uint8, device="cuda")])
    b.sync()
    prof = b.profile_read()[0]
    b.close()
    # one launch from the packed samples, and none that unpacks them first
    assert prof["xengine"]["launches"] == 1 and prof["unpack"]["launches"] == 0
