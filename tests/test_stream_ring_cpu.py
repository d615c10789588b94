"""The streaming solve's shared memory: one layout serves every subdomain of a handle, from the
largest of each part, so the ring of panels has to keep its three stages for any mixture of
subdomains that the rule admits, not only for each one by itself."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda/include"

SOURCE = r"""
#include <cstdio>
#include "mrcm_internal.h"
int main() {
    mrcm::BigSmem all;
    int n = 0, least = 99;
    for (int b = 1; b <= mrcm::kMaxBlock; ++b)
        for (int m = 1; m <= 2 * mrcm::kMaxI + 1; ++m)
            if (mrcm::big_ok(b, m)) {
                mrcm::BigSmem one;
                one.add(b, m);
                all.add(b, m);
                least = one.stages() < least ? one.stages() : least;
                ++n;
            }
    std::printf("%d %d %d %zu %zu", n, least, all.stages(), all.total(), mrcm::kSolveSmemBudget);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.isdir(CUDA), reason="needs g++ and the CUDA headers")
def test_ring_of_any_mixture_of_subdomains(tmp_path):
    src = tmp_path / "ring.cpp"
    src.write_text(SOURCE)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2103_08513_gb300", "csrc"), "-I",
                           os.path.join(ROOT, "include"), "-I", CUDA, str(src), "-o", str(tmp_path / "ring")])
    n, least, together, total, budget = map(int, subprocess.check_output([str(tmp_path / "ring")]).split())
    assert n > 10000 and least >= 3 and together >= 3 and total <= budget
