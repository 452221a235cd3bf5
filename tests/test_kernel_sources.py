"""Instruction forms that the kernels' sources must not use."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1501_05992_gb300", "csrc")


def test_no_copy_is_multicast_over_a_cluster():
    """One libcorr.so serves every rank of a job on several GPUs, on whatever buffer the caller
    passes, and loads multicast over a cluster are for code of one GPU only (a barrier arrival by
    tcgen05.commit is no load)."""
    for path in glob.glob(os.path.join(CSRC, "*")):
        if os.path.isfile(path):
            with open(path) as f:
                text = re.sub(r'"\s*"', "", f.read())
            for op in re.findall(r"cp\.async\.bulk[\w.:]*", text):
                assert "multicast" not in op, (os.path.basename(path), op)
