"""Host-side check of how a layer on host buffers divides its batch (psa_sched.h compiled with g++)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "paper_2012_01114_b200/csrc/psa_sched.h"
int main(int argc, char** argv) {
    unsigned long long a[5];
    for (int i = 0; i < 5; ++i) a[i] = strtoull(argv[i + 1], nullptr, 0);
    printf("%d\n", psa::host_parts((int)a[0], a[1], a[2], (const void*)a[3], (const void*)a[4]));
    return 0;
}
"""


@pytest.fixture(scope="module")
def parts(tmp_path_factory):
    d = tmp_path_factory.mktemp("parts")
    src = d / "parts.cpp"
    src.write_text(SRC)
    exe = d / "parts"
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", ROOT, "-o", str(exe), str(src)])
    return lambda *a: int(subprocess.check_output([str(exe)] + [str(x) for x in a]))


X = 1 << 32


# 8 sequences of 1 MB in and 2 MB out: 8 parts as long as the buffers are apart, one as soon as a single byte is shared
@pytest.mark.parametrize("out,want", [(X + (8 << 20), 8), (X + (8 << 20) - 1, 1), (X, 1), (X - (16 << 20), 8),
                                      (X - (16 << 20) + 1, 1), (X - (4 << 20), 1), (X + (1 << 20), 1)])
def test_overlapping_buffers_go_in_one_part(parts, out, want):
    assert parts(8, 1 << 20, 2 << 20, X, out) == want


@pytest.mark.parametrize("batch,x,out,want", [(1, 1 << 30, 1 << 30, 1), (8, 1 << 10, 1 << 10, 1), (4, 1 << 20, 1 << 20, 2),
                                              (100, 1 << 20, 1 << 20, 8), (3, 4 << 20, 4 << 20, 3)])
def test_parts_of_separate_buffers(parts, batch, x, out, want):
    assert parts(batch, x, out, X, 1 << 50) == want
