"""Host-side check of the workspace's layout (psa_ws.h compiled with g++): nothing overlaps, and what a part of a host call takes for its projections
lies in the room that the layout of the whole call has for it.  And which memory a call runs in, the lean layout of fp32 calls included."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <utility>
#include <vector>
#include "paper_2012_01114_b200/csrc/psa_ws.h"
using namespace psa;
typedef std::pair<size_t, size_t> Range;       // first byte, bytes

static std::vector<Range> ranges(const WsShape& c, const WsLayout& L) {
    const size_t es = c.dtype == PSA_BF16 ? 2 : 4, rows = (size_t)c.batch * c.n, hd = (size_t)c.heads * c.d_k, bh = (size_t)c.batch * c.heads;
    const size_t in = rows * c.d_model * es, w = (size_t)c.d_model * hd * es, qkv = rows * hd * es;
    std::vector<Range> r{{0, COUNTER_BYTES}};
    size_t parts = L.in_bytes > L.out_bytes ? L.in_bytes : L.out_bytes;
    if (L.attn_tensor) {
        r.push_back({L.bad, bh * 4});
        r.push_back({L.ml, 2 * bh * c.n * 4});
        if (parts < 12 * rows * hd) parts = 12 * rows * hd;
    }
    if (L.in_bytes) r.push_back({L.marks_in, f32_project_marks((int)rows, (int)hd, 3) * 4 * (c.staging ? HOST_CHUNKS : 1)});
    if (L.out_bytes) r.push_back({L.marks_out, f32_project_marks((int)rows, c.d_model, 1) * 4});
    if (parts) r.push_back({L.parts, parts});
    const bool sym = c.scheme == PSA_SYMMETRIC;
    if (sym) r.push_back({L.s, L.s_bytes});
    if (c.with_proj) { r.push_back({L.q, qkv}); if (!sym) { r.push_back({L.k, qkv}); r.push_back({L.v, qkv}); } }
    if (c.staging) {
        r.push_back({L.xs, in}); r.push_back({L.wq, w}); r.push_back({L.outs, qkv});
        if (!sym) { r.push_back({L.wk, w}); r.push_back({L.wv, w}); }
    }
    return r;
}

int main() {
    // the last three: X of 2^33 numbers and more, with and without room for the parts of an output projection
    const int shapes[][5] = {{1, 1, 64, 64, 64}, {4, 12, 512, 768, 64}, {9, 5, 300, 328, 40}, {64, 16, 1024, 128, 128}, {33, 1, 1023, 2048, 8}, {3, 7, 1, 24, 20},
                             {2100, 33, 1, 776, 32}, {1024, 4, 1024, 8192, 64}, {1030, 1, 1024, 8192, 8}, {1100, 16, 1024, 8192, 128}};
    long long used = 0, refused = 0;
    for (const auto& s : shapes)
        for (int scheme : {PSA_FULL, PSA_SYMMETRIC, PSA_MASKED})
            for (int dtype : {PSA_F32, PSA_BF16})
                for (int kind = 0; kind < 4; ++kind) {
                    const WsShape c{s[0], s[1], s[2], kind ? s[3] : 0, s[4], scheme, dtype, kind > 0, kind > 1, kind == 3, false};
                    const WsLayout L = ws_layout(c);
                    WsShape lean = c;
                    lean.lean = true;
                    const WsLayout M = ws_layout(lean);
                    // lean: counters, scores, q, k, v and staging only, all that the CUDA cores need
                    size_t rest = COUNTER_BYTES;
                    for (const Range& x : ranges(lean, M)) rest += x.first ? align_up(x.second, 256) : 0;
                    if (M.total != rest || M.attn_tensor || M.in_bytes || M.out_bytes || M.clear_bytes) return 6;
                    if (M.total > L.total || (dtype == PSA_BF16 && M.total != L.total)) return 7;
                    const std::vector<Range> r = ranges(c, L);
                    for (size_t i = 0; i < r.size(); ++i) {
                        if (r[i].first % 256 || r[i].first + r[i].second > L.total) return 2;
                        for (size_t j = 0; j < i; ++j)
                            if (r[i].first < r[j].first + r[j].second && r[j].first < r[i].first + r[i].second) return 3;
                    }
                    if (dtype != PSA_F32 || kind != 2) continue;
                    const int nW = scheme == PSA_SYMMETRIC ? 1 : 3, hd = c.heads * c.d_k;
                    for (int parts = 1; parts <= HOST_CHUNKS && parts <= c.batch; ++parts)
                        for (int k = 0; k < parts; ++k) {
                            const int nb = (int)((long long)c.batch * (k + 1) / parts - (long long)c.batch * k / parts);
                            const size_t need = f32_project_parts_bytes(nb * c.n, c.d_model, hd, nW);
                            if (!need) continue;
                            if (!f32_project_pairs_fit(nb * c.n, c.d_model, hd, nW, L.in_bytes)) { ++refused; continue; }
                            ++used;
                            if (need > L.in_bytes) return 4;
                            // marks of part k: behind those of the part before, before those of the next
                            if (f32_project_marks(nb * c.n, hd, nW) > L.marks_pitch) return 5;
                            const size_t last = L.marks_in + (k * L.marks_pitch + f32_project_marks(nb * c.n, hd, nW)) * 4;
                            if (L.marks_in < L.clear || last > L.clear + L.clear_bytes || (L.marks_out && L.marks_in < L.marks_out && last > L.marks_out)) return 8;
                        }
                }
    printf("%lld %lld\n", used, refused);
    return 0;
}
"""


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    (d / "layout.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", ROOT, "-o", str(d / "layout"), str(d / "layout.cpp")])
    return str(d / "layout")


def test_nothing_overlaps_and_parts_stay_inside(layout):
    run = subprocess.run([layout], capture_output=True, text=True)
    assert run.returncode == 0, run.returncode
    used, refused = (int(x) for x in run.stdout.split())
    assert used > 20 and refused > 20        # parts of calls with and without room


PLAN = r"""
#include <cstdio>
#include <cstdlib>
#include "paper_2012_01114_b200/csrc/psa_ws.h"
int main(int, char** a) {
    bool asked = false;
    const psa::WsPlan p = psa::ws_plan(atoi(a[1]), atoi(a[2]), atoi(a[3]), atoi(a[4]), [&] { asked = true; return atoi(a[5]) != 0; });
    printf("%d %d %d\n", (int)p.from, (int)p.whole, (int)asked);
    return 0;
}
"""
USER, OWN, GROW = 0, 1, 2


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(PLAN)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", ROOT, "-o", str(d / "plan"), str(d / "plan.cpp")])
    return lambda *a: tuple(int(x) for x in subprocess.check_output([str(d / "plan")] + [str(x) for x in a]).split())


# bytes registered, of the library's own workspace, of the whole layout, of the lean one; whether there is memory to grow into
@pytest.mark.parametrize("user,own,whole,least,memory,want", [
    (100, 0, 100, 40, 0, (USER, 1, 0)), (99, 100, 100, 40, 1, (USER, 0, 0)), (40, 0, 100, 40, 1, (USER, 0, 0)), (39, 100, 100, 40, 0, (OWN, 1, 0)),
    (39, 99, 100, 40, 0, (OWN, 0, 1)), (0, 40, 100, 40, 0, (OWN, 0, 1)), (0, 40, 100, 40, 1, (GROW, 1, 1)), (0, 39, 100, 40, 0, (GROW, 1, 0)),
    (0, 0, 100, 40, 0, (GROW, 1, 0)), (0, 99, 100, 100, 0, (GROW, 1, 0)), (99, 100, 100, 100, 0, (OWN, 1, 0))])
def test_memory_of_a_call(plan, user, own, whole, least, memory, want):
    assert plan(user, own, whole, least, memory) == want


FITS = r"""
#include <cstdio>
#include <cstdlib>
#include "paper_2012_01114_b200/csrc/psa_ws.h"
int main(int argc, char** a) {
    for (int i = 1; i + 4 < argc; i += 5)
        printf("%d ", (int)psa::f32_tensor_attention_fits(atoi(a[i]), atoi(a[i + 1]), atoi(a[i + 2]), atoi(a[i + 3]), atoi(a[i + 4])));
    return 0;
}
"""
FULL, MASKED = 0, 2


def test_calls_with_little_off_the_diagonal_tiles_stay_on_cuda_cores(tmp_path):
    # (batch, heads, n, d, scheme) measured faster on CUDA cores, and neighbours measured faster on the tensor cores
    cuda = [(1, 29, 257, 64, MASKED), (2, 16, 257, 64, MASKED), (1, 29, 257, 128, MASKED), (1, 53, 257, 128, MASKED), (1, 48, 257, 16, MASKED), (1, 29, 300, 64, MASKED),
            (4, 14, 320, 64, MASKED), (1, 53, 320, 8, MASKED), (1, 123, 320, 8, MASKED), (1, 16, 385, 64, MASKED), (4, 5, 385, 64, MASKED), (1, 22, 385, 32, MASKED),
            (1, 20, 385, 8, MASKED), (1, 20, 420, 64, MASKED), (1, 17, 513, 8, MASKED), (1, 8, 257, 16, FULL), (1, 17, 256, 8, FULL)]
    tensor = [(1, 64, 257, 64, MASKED), (1, 40, 257, 128, MASKED), (1, 64, 300, 64, MASKED), (1, 32, 300, 64, MASKED), (1, 79, 320, 64, MASKED), (1, 24, 385, 64, MASKED),
              (4, 6, 385, 32, MASKED), (1, 20, 513, 8, MASKED), (1, 4, 1024, 64, MASKED), (2, 8, 1024, 128, MASKED), (1, 8, 257, 32, FULL), (1, 12, 257, 8, FULL),
              (1, 20, 256, 8, FULL), (1, 1, 1024, 8, FULL), (4, 12, 512, 64, FULL)]
    (tmp_path / "fits.cpp").write_text(FITS)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", ROOT, "-o", str(tmp_path / "fits"), str(tmp_path / "fits.cpp")])
    got = subprocess.check_output([str(tmp_path / "fits")] + [str(x) for c in cuda + tensor for x in c]).split()
    assert [int(x) for x in got] == [0] * len(cuda) + [1] * len(tensor)


MARKS = r"""
#include <cstdio>
#include "paper_2012_01114_b200/csrc/psa_ws.h"
using namespace psa;
int main() {
    // a block whose layer runs in one launch, and one whose layer does not: marks behind the counters, all in the range that a captured call clears
    for (bool one_launch : {true, false}) {
        const WsLayout L = ws_layout(WsShape{400, 16, 64, 256, 16, PSA_FULL, PSA_F32, true, false, one_launch, false});
        const size_t marks = f32_project_marks(400 * 64, 256, 1) * sizeof(int);
        if (!L.out_bytes || L.clear != COUNTER_BYTES || L.marks_out < L.clear || L.marks_out + marks > L.clear + L.clear_bytes) return 1;
    }
    return 0;
}
"""


def test_marks_of_an_output_projection_lie_in_what_a_captured_call_clears(tmp_path):
    (tmp_path / "marks.cpp").write_text(MARKS)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", ROOT, "-o", str(tmp_path / "marks"), str(tmp_path / "marks.cpp")])
    assert subprocess.call([str(tmp_path / "marks")]) == 0
