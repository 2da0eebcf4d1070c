"""Host-side check of how a layer on host buffers divides its batch, and of the symmetric scheme's passes over the heads of a
part (psa_sched.h compiled with g++)."""
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


PASSES = r"""
#include <cstdio>
#include <cstdlib>
#include "paper_2012_01114_b200/csrc/psa_sched.h"
using namespace psa;
// Heads per pass of a whole call and of its parts, which share the scratch that the whole call is given.
int main() {
    const int lengths[] = {1, 128, 129, 1000, 2048, 3001, 4096, 7296, 8192, 16384, 40000, 100000};
    const int head_counts[] = {1, 2, 3, 4, 5, 8, 12, 16, 20, 32};
    long long cases = 0, less = 0;
    for (int n : lengths) {
        const size_t per_head = (size_t)sym_pairs(row_tiles(n)) * S_BLOCK_BYTES;
        for (int H : head_counts)
            for (int B = 1; B <= 260; ++B) {
                const int whole = sym_heads_per_pass((size_t)B * H, n, SYM_SCRATCH_CAP);
                if (whole < 1 || whole > B * H || (whole > 1 && whole * per_head > SYM_SCRATCH_CAP)) return 2;
                if (sym_heads_per_pass((size_t)B * H, n, whole * per_head) != whole) return 3;
                for (int parts = 2; parts <= HOST_CHUNKS && parts <= B; ++parts)
                    for (int nb = B / parts; nb <= (B + parts - 1) / parts; ++nb, ++cases) {
                        const int hp = sym_heads_per_pass((size_t)nb * H, n, whole * per_head);
                        if (hp < 1 || hp > whole || hp > nb * H) return 4;
                        less += hp < sym_heads_per_pass((size_t)nb * H, n, SYM_SCRATCH_CAP);
                    }
            }
    }
    printf("%lld %lld\n", cases, less);
    return 0;
}
"""


def test_passes_of_a_part_fit_the_scratch_of_the_call(tmp_path):
    src = tmp_path / "passes.cpp"
    src.write_text(PASSES)
    exe = tmp_path / "passes"
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", ROOT, "-o", str(exe), str(src)])
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.returncode
    cases, less = (int(x) for x in run.stdout.split())
    assert cases > 100000 and less > 100         # parts that alone would take more heads per pass than the whole call
