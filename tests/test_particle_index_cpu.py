"""Tile walks near the largest particle count (no GPU needed).

A run takes up to 2^31 - 1 particles, and a walk looks one stride ahead of its particle.
The walk's index type is compiled for the host and stepped past the last particles at
every block size; the kernels' walks are held to that type.
"""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_11052_gb300", "csrc")

PROGRAM = r"""
#include "pic_internal.cuh"
#include <cstdio>
int main() {
    const long long most = 2147483647ll;
    for (unsigned step : {64u, 256u, 384u, 1024u})
        for (long long first : {most - 1ll, most - 63ll, most - 5000ll}) {
            const pic::PIndex begin = (pic::PIndex)first, end = (pic::PIndex)most;
            long long seen = 0, ahead = 0;
            for (unsigned t = 0; t < step; ++t) {
                pic::PIndex p = begin + t;
                for (int turn = 0; p < end; p += step, ++turn) {
                    if (turn > 5000 || (long long)p < first || (long long)p >= most) return 1;
                    ++seen;
                    const pic::PIndex pn = p + step;
                    if (pn < end) {
                        if ((long long)pn >= most || (long long)pn <= first) return 2;
                        ++ahead;
                    }
                }
            }
            const long long n = most - first;
            if (seen != n || ahead != (n > (long long)step ? n - (long long)step : 0)) return 3;
        }
    std::puts("ok");
    return 0;
}
"""


def test_a_walk_ends_at_the_largest_count(tmp_path):
    from paper_2205_11052_gb300.build import ARCH, _nvcc

    nvcc = _nvcc()
    if not shutil.which(nvcc) and not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    src = tmp_path / "walk.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "walk")
    subprocess.run([nvcc, *ARCH, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", exe],
                   check=True, capture_output=True)
    assert subprocess.run([exe], capture_output=True, text=True).stdout.strip() == "ok"


def test_walks_use_that_type():
    walks = 0
    for f in glob.glob(os.path.join(CSRC, "k_*.cu")):
        text = open(f).read()
        walks += len(re.findall(r"PIndex p = \w+(?:\.y)? \+ threadIdx\.x", text))
        assert not re.search(r"\bint (?:p|pn) = (?:begin|item\.y|p) \+", text), f
    assert walks == 6      # push, move, deposit (dense and sparse), reverse push, batched push
