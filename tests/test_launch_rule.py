"""The rule that sizes the persistent kernel's grid (host code of
svt_internal.h, compiled here)."""
import os
import subprocess

import pytest

from paper_1312_0917_gb300 import build

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "svt_internal.h"
int main(int, char **a)
{
    std::printf("%d", svt::ctas_per_sm(std::atoll(a[1]), 152, std::atoi(a[2]), std::atoi(a[3]), std::atoi(a[4])));
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    if not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    d = tmp_path_factory.mktemp("rule")
    src, exe = str(d / "rule.cpp"), str(d / "rule")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-I" + build.CSRC, "-I" + build.INCLUDE, "-I" + cuda, src, "-o", exe])
    return lambda *a: int(subprocess.check_output([exe] + [str(x) for x in a]))


@pytest.mark.parametrize("block,most", [(128, 6), (256, 3), (512, 1)])
def test_ctas_per_sm(rule, block, most):
    """Settings below the maximum as given; 0 and the maximum, which is how 0
    reads back, both by the words, on either side of each line."""
    for words in (0, 1, 640 * 152, 640 * 152 + 1, 3072 * 152, 3072 * 152 + 1, 1 << 30):
        by_words = rule(words, block, most, 0)
        threads = 256 if words <= 640 * 152 else 512 if words <= 3072 * 152 else 1 << 20
        assert by_words == min(max(threads // block, 1), most)
        assert rule(words, block, most, most) == rule(words, block, most, most + 5) == by_words
        for few in range(1, most):
            assert rule(words, block, most, few) == few
