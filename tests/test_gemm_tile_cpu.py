"""Which output tile a bf16 projection takes (psa_sched.h compiled with g++): M rows, K deep, nW matrices of N columns."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "paper_2012_01114_b200/csrc/psa_sched.h"
int main(int argc, char** a) {
    for (int i = 1; i + 3 < argc; i += 4) printf("%d ", (int)psa::gemm_tile(atoi(a[i]), atoi(a[i + 1]), atoi(a[i + 2]), atoi(a[i + 3]), 148));
    return 0;
}
"""
LONE_128, LONE_192, LONE_256, PAIR_256 = range(4)


def _tiles(tmp_path, calls):
    (tmp_path / "tile.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", ROOT, "-o", str(tmp_path / "tile"), str(tmp_path / "tile.cpp")])
    return [int(x) for x in subprocess.check_output([str(tmp_path / "tile")] + [str(x) for c in calls for x in c]).split()]


def test_sizes_measured_on_either_side(tmp_path):
    want = {
        # faster on 192 columns
        (2048, 768, 512, 3): LONE_192, (4096, 768, 576, 3): LONE_192, (8192, 256, 576, 3): LONE_192, (8192, 3072, 576, 3): LONE_192, (16384, 192, 320, 3): LONE_192,
        (8192, 768, 768, 1): LONE_192, (19328, 3072, 576, 3): LONE_192, (60032, 384, 384, 3): LONE_192, (9088, 2048, 576, 3): LONE_192,
        # long runs that are faster on pairs
        (640, 2560, 2560, 3): PAIR_256, (768, 2560, 2560, 3): PAIR_256, (1280, 2560, 2560, 3): PAIR_256, (1024, 2048, 2048, 3): PAIR_256, (4096, 3072, 512, 3): PAIR_256,
        (3072, 3072, 768, 3): PAIR_256, (7040, 4096, 768, 1): PAIR_256, (54144, 768, 192, 3): PAIR_256, (32768, 1536, 192, 3): PAIR_256,
        # sizes at which 192 columns take more rounds, or leave SMs idle
        (8192, 768, 768, 3): PAIR_256, (4096, 768, 768, 3): LONE_256, (200, 768, 768, 3): LONE_128, (4096, 1536, 384, 3): LONE_128}
    assert dict(zip(want, _tiles(tmp_path, list(want)))) == want


def test_sizes_of_the_gpu_tests(tmp_path):
    # the sizes of test_projections_on_tiles_of_192_columns and test_layers_on_tiles_of_192_columns (tests/test_gpu_block.py)
    calls = [(2048, 512, 512, 3), (1990, 576, 512, 3), (4000, 512, 192, 3), (2700, 512, 320, 3), (1000, 512, 1024, 3), (4090, 768, 768, 1),
             (2000, 576, 512, 3), (2709, 512, 320, 3), (8000, 512, 704, 1)]
    assert _tiles(tmp_path, calls) == [LONE_192] * len(calls)
