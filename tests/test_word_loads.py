"""The channels whose words the any-byte loads of the tensor-core X-engine test against the
array's ends: every other channel's words lie within the array, on every byte offset of its
buffer (computed on the host, from the function that the kernel uses)."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include "internal.cuh"
extern "C" int reach_over(int f, int n_chan, int n) { return corr::words_reach_over(f, n_chan, n); }
"""


@pytest.fixture(scope="module")
def reach_over(tmp_path_factory):
    d = tmp_path_factory.mktemp("words")
    src, lib = d / "words.cpp", d / "words.so"
    src.write_text(SOURCE)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    inc = [os.path.join(ROOT, "paper_1501_05992_gb300", "csrc"), os.path.join(ROOT, "include"), cuda,
           "/usr/local/cuda/include"]
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", str(src), "-o", str(lib)] + [f"-I{i}" for i in inc],
                   check=True)
    return ctypes.CDLL(str(lib)).reach_over


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 130, 250])
@pytest.mark.parametrize("n_chan", [1, 2, 3, 4, 5, 8])
def test_words_of_other_channels_lie_within(reach_over, n, n_chan):
    for offset in range(4):                       # of the buffer from a word boundary
        for n_time in (1, 2, 3):
            lo, hi = offset, offset + n_time * n_chan * n
            for t in range(n_time):
                for f in range(n_chan):
                    first = offset + (t * n_chan + f) * n
                    begin, end = first // 4 * 4, (first + n + 3) // 4 * 4
                    assert reach_over(f, n_chan, n) or (begin >= lo and end <= hi), (offset, n_time, t, f)


def test_inner_channels_of_ordinary_rows_are_not_tested(reach_over):
    assert [f for f in range(768) if reach_over(f, 768, 250)] == [0, 767]
