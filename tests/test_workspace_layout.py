"""The workspace of the block-tiled reverse pass (csrc/tile_layout.h): no more than the call can use, within the bound it states."""
import pathlib
import subprocess

from paper_2608_21308_b200 import binding as E

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2608_21308_b200" / "csrc"

LAYOUTS = r"""
#include "simt_layout.h"
#include <cstdio>
#include <initializer_list>
using namespace e2ttt;
int main() {
    int bad = 0;
    for (int N : {1, 4, 16, 32, 33, 34, 64, 150, 2048})
        for (int d : {8, 64, 128})
            for (int h : {8, 192, 512, 1024, 1088})
                for (int C : {16, 64, 65, 512})
                    for (int nmat : {2, 3})
                        for (int nchunks : {1, 2, 3, 8, 23, 128})
                            for (int seg : {0, 2, 4, 32}) {
                                const SimtLayout l = simt_layout(d, h, C, nmat, nchunks, true, true, seg, 1, N);
                                const TileLayout& t = l.tl;
                                const int chunks = seg > 0 && seg < nchunks ? seg : nchunks;
                                const size_t slots = (size_t)t.G * N * t.slot_stride * 4, one = (size_t)N * t.slot_stride * 4;
                                const bool unused = t.G > chunks || (t.sets == 2 && chunks <= t.G);
                                const bool over = slots > (one > ((size_t)512 << 20) ? one : (size_t)512 << 20);
                                const bool outside = t.slot + (size_t)t.sets * t.G * t.slot_stride > l.per_seq;
                                if ((unused || over || outside || t.G < 1) && bad++ < 5)
                                    std::printf("N=%d d=%d h=%d C=%d nmat=%d chunks=%d: G=%d sets=%d\n", N, d, h, C, nmat, chunks, t.G, t.sets);
                            }
    return bad != 0;
}
"""


def test_slots_of_the_reverse_pass_are_bounded_by_the_chunks_of_a_launch(tmp_path):
    (tmp_path / "layouts.cpp").write_text(LAYOUTS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(CSRC), str(tmp_path / "layouts.cpp"), "-o", str(tmp_path / "layouts")], check=True)
    out = subprocess.run([str(tmp_path / "layouts")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


def test_a_short_training_call_asks_for_one_chunks_slots():
    """16 sequences of one chunk, d = 128, h = 512: 9.0 MB each, of which one slot is 1.83 MB (16 slots would make it 36.4 MB)."""
    p = E.make_params(1, 16, 64, 128, 512, 64, E.E2TTT_MLP_GELU, E.E2TTT_BF16, 1e-5, E.E2TTT_IMPL_AUTO)
    assert E.e2ttt_workspace_bytes(p, 1) < 16 * 9.5e6


F64 = r"""
#include "simt_layout.h"
#include <initializer_list>
using namespace e2ttt;
int main() {
    for (int N : {1, 13, 64, 2048})
        for (int d : {1, 64, 128, 1024})
            for (int h : {1, 256, 8192})
                for (int C : {1, 16, 64, 512})
                    for (int nmat : {2, 3})
                        for (int nchunks : {1, 5, 300})
                            for (int seg : {0, 4}) {
                                const SimtLayout l = simt_layout(d, h, C, nmat, nchunks, true, true, seg, 0, N, 1);
                                const F64Layout& f = l.fl;
                                const int chunks = seg > 0 && seg < nchunks ? seg : nchunks;
                                if (f.G < 1 || f.G > chunks) return 1;
                                if (f.G > 1 && f.slot_stride * 8 * f.G * N > kF64SlotBytes) return 2;
                                if (f.slot + f.slot_stride * f.G > l.per_seq) return 3;
                            }
    return 0;
}
"""


def test_slots_of_the_fp64_reverse_pass_are_bounded(tmp_path):
    (tmp_path / "f64.cpp").write_text(F64)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(CSRC), str(tmp_path / "f64.cpp"), "-o", str(tmp_path / "f64")], check=True)
    assert subprocess.run([str(tmp_path / "f64")]).returncode == 0


def test_slots_stop_where_more_of_them_do_not_pay():
    """fp32, one sequence of 4096 tokens in chunks of 16, d = 64, h = 256: 256 chunks, of which 148 are prepared at a time (187 MB; the 64 MB
    that slots may take would make it 195).  64 sequences of chunks of one token, d = h = 16: 32 MB of slots."""
    mb = lambda *a: E.e2ttt_workspace_bytes(E.make_params(*a, E.E2TTT_MLP_GELU, E.E2TTT_F32, 1e-5, E.E2TTT_IMPL_AUTO), 1) / 2**20
    assert 185 < mb(1, 1, 4096, 64, 256, 16) < 189
    assert mb(64, 1, 256, 16, 16, 1) < 170
    assert mb(1, 1, 256, 64, 256, 16) < 16
