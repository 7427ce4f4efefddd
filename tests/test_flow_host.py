"""The forward on work items, host side (csrc/tile_flow.h): the queue hands out every item once and after those it depends on; which calls take it."""
import pathlib
import subprocess

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2608_21308_b200" / "csrc"


def run(tmp_path, source):
    (tmp_path / "t.cpp").write_text("#include <cstdio>\n#include <initializer_list>\n#include <vector>\n#include \"tile_flow.h\"\nusing namespace e2ttt;\n" + source)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", str(CSRC), str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")], check=True)
    out = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout


QUEUE = r"""
int several_last_short = 0, shifted = 0;
bool check(int N, int d, int h, int C, int L, int nmat, bool normed) {
    TileLayout tl{};
    tl.db = (d + 63) / 64; tl.hb = (h + 63) / 64; tl.tb = (C + 63) / 64;
    const FlowPlan f = flow_plan(tl, N, L, C, nmat, normed);
    if (f.sets > 1 && f.sets * f.gs > N) ++several_last_short;
    if (f.off2 > 0) ++shifted;
    if ((long long)f.sets * f.gs < N || f.gs < 1) return false;
    std::vector<int> tokens(N), weights(N), norms(N);  // done so far, as the kernel counts them
    std::vector<char> seen((size_t)N * f.nchunks * f.slots);
    for (long long id = 0;; ++id) {
        const FlowItem it = flow_item(f, id);
        if (it.type == kFlowEnd) break;
        if (it.type == kFlowNone) continue;
        if (it.seq < 0 || it.seq >= N || it.c < 0 || it.c >= f.nchunks) return false;
        const int len = L - it.c * C < C ? L - it.c * C : C, blocks = (len + 63) / 64;
        int slot = it.part;
        if (it.type == kFlowTokens) {
            if (it.part >= blocks || (normed ? norms : weights)[it.seq] < it.c * (normed ? f.n3 : f.n2)) return false;
            ++tokens[it.seq];
        } else if (it.type == kFlowWeights) {
            if (it.part >= f.n2 || tokens[it.seq] < it.c * tl.tb + blocks) return false;
            ++weights[it.seq];
            slot += f.tb;
        } else {
            if (it.part >= f.n3 || weights[it.seq] < (it.c + 1) * f.n2) return false;
            ++norms[it.seq];
            slot += f.tb + f.n2;
        }
        char& once = seen[((size_t)it.seq * f.nchunks + it.c) * f.slots + slot];
        if (once++) return false;
    }
    const int blocks = (L / C) * ((C + 63) / 64) + (L % C + 63) / 64;
    for (int s = 0; s < N; ++s)
        if (tokens[s] != blocks || weights[s] != f.nchunks * f.n2 || norms[s] != f.nchunks * f.n3) return false;
    return true;
}
int main() {
    for (int N : {1, 2, 15, 16, 37, 67, 101, 150, 257})
        for (int d : {8, 128})
            for (int h : {8, 384, 520, 1100, 8192})
                for (int C : {1, 24, 64, 65, 200, 512})
                    for (int L : {1, 63, 64, 65, 300, 1100})
                        for (int nmat : {2, 3})
                            for (int normed = 0; normed < 2; ++normed)
                                if (!(C == 1 && L > 65) && !(h == 8192 && (L > 300 || C < 24 || N > 101)) && !check(N, d, h, C, L, nmat, normed)) {
                                    std::printf("N=%d d=%d h=%d C=%d L=%d nmat=%d normed=%d\n", N, d, h, C, L, nmat, normed);
                                    return 1;
                                }
    return several_last_short > 100 && shifted > 100 ? 0 : 2;
}
"""


def test_the_queue_hands_out_every_item_once_and_in_order(tmp_path):
    run(tmp_path, QUEUE)


LINES = r"""
struct Call { int N, d, h, C, L, nmat; bool flow, normed = false; };
int main() {
    int bad = 0;
    auto flow = [](const Call& c, int Ls) {
        TileLayout tl{};
        tl.db = (c.d + 63) / 64; tl.hb = (c.h + 63) / 64; tl.tb = (c.C + 63) / 64;
        return tile_flow_serves(tl, c.N, c.C, Ls, c.nmat, c.normed);
    };
    for (const Call& c : {  // calls that were measured on both kernels, and the faster one
             // shorter than their chunk: the blocks that they have count, not the chunk's
             Call{1, 128, 2048, 512, 64, 2, false}, Call{8, 128, 1024, 512, 64, 2, false}, Call{8, 128, 1024, 512, 128, 2, false}, Call{8, 128, 1024, 512, 192, 2, true},
             Call{15, 128, 2048, 512, 64, 2, false}, Call{20, 128, 2048, 512, 64, 2, false}, Call{8, 128, 1024, 512, 512, 2, true}, Call{64, 128, 512, 512, 64, 2, true},
             // one chunk
             Call{33, 64, 448, 64, 64, 2, false}, Call{16, 64, 640, 64, 64, 2, false}, Call{64, 128, 640, 64, 64, 2, true}, Call{15, 128, 384, 64, 64, 3, true},
             // wide networks, several chunks of one block
             Call{16, 128, 8192, 64, 128, 2, false}, Call{22, 64, 4096, 16, 64, 2, false}, Call{20, 128, 768, 64, 512, 2, true}, Call{24, 128, 1024, 64, 512, 2, true},
             Call{16, 128, 768, 64, 512, 3, true}, Call{8, 128, 1024, 64, 512, 2, false}, Call{8, 128, 384, 64, 512, 2, true}, Call{8, 128, 1024, 128, 512, 2, false},
             Call{16, 128, 1024, 128, 512, 2, true}, Call{64, 128, 512, 512, 2048, 2, true},
             // normalised
             Call{33, 64, 2048, 64, 256, 3, false, true}, Call{33, 64, 2048, 64, 256, 3, true}, Call{64, 128, 2048, 128, 512, 3, false, true},
             Call{8, 128, 384, 64, 256, 2, false, true}, Call{16, 128, 384, 64, 256, 3, true, true}, Call{33, 128, 2048, 512, 1024, 2, true, true}})
        if (flow(c, c.L) != c.flow && bad++ < 9) std::printf("N=%d d=%d h=%d C=%d L=%d nmat=%d\n", c.N, c.d, c.h, c.C, c.L, c.nmat);
    return bad != 0;
}
"""


def test_calls_take_the_kernel_that_measured_the_faster(tmp_path):
    run(tmp_path, LINES)


SPLIT = r"""
int main() {
    for (int N : {1, 2, 8, 15, 16, 19, 22, 23, 25, 33, 34, 64, 75, 148})
        for (int d : {64, 128})
            for (int hb = 1; hb <= 80; ++hb)
                for (int C : {16, 64, 100, 128, 192, 256, 512})
                    for (int nmat : {2, 3})
                        for (int normed = 0; normed < 2; ++normed) {
                            TileLayout tl{};
                            tl.db = d / 64; tl.hb = hb; tl.tb = (C + 63) / 64;
                            const bool one = tile_flow_serves(tl, N, C, C, nmat, normed);
                            for (int Ls : {C + 1, 2 * C, 4 * C, 31 * C + 3})
                                if (tile_flow_serves(tl, N, C, Ls, nmat, normed) != one) {
                                    std::printf("N=%d d=%d hb=%d C=%d Ls=%d nmat=%d normed=%d\n", N, d, hb, C, Ls, nmat, normed);
                                    return 1;
                                }
                        }
    return 0;
}
"""


def test_a_sequence_in_several_calls_takes_the_kernel_of_one(tmp_path):
    run(tmp_path, SPLIT)


FIRST = r"""
int main() {
    int few = 0;
    for (int N : {1, 5, 34, 64, 74, 100, 148, 149})
        for (int h : {64, 192, 512})
            for (int C : {16, 64, 128, 512})
                for (int nmat : {2, 3})
                    for (int normed = 0; normed < 2; ++normed) {
                        TileLayout tl{};
                        tl.db = 2; tl.hb = h / 64; tl.tb = (C + 63) / 64;
                        const FlowPlan f = flow_plan(tl, N, C, C, nmat, normed);
                        if (N * f.tb > 148 || N * f.slots <= 148) continue;
                        ++few;
                        long long tokens = 0, id = 0;
                        for (FlowItem it = flow_item(f, 0); it.type != kFlowEnd; it = flow_item(f, ++id)) {
                            if (it.type == kFlowTokens) ++tokens;
                            if (it.type == kFlowWeights && tokens < (long long)N * f.tb) {
                                std::printf("N=%d h=%d C=%d nmat=%d normed=%d\n", N, h, C, nmat, normed);
                                return 1;
                            }
                        }
                    }
    return few > 40 ? 0 : 2;
}
"""


def test_single_chunks_start_with_their_tokens(tmp_path):
    run(tmp_path, FIRST)


PADDING = r"""
struct Call { int N, d, h, C; bool off; };
int main() {
    int bad = 0;
    for (const Call& c : {  // calls of one and of four chunks were measured on both kernels; the faster one (where the two differ: over both)
             Call{148, 8, 8, 1, true}, Call{148, 64, 64, 4, true}, Call{148, 64, 72, 4, true}, Call{148, 40, 104, 1, true}, Call{148, 32, 160, 4, true}, Call{148, 16, 300, 1, true},
             Call{148, 8, 600, 1, true}, Call{120, 64, 64, 1, true}, Call{100, 16, 16, 4, true}, Call{100, 32, 32, 1, true}, Call{296, 64, 64, 1, true}, Call{296, 16, 300, 4, true},
             Call{590, 16, 16, 16, true}, Call{592, 64, 64, 4, true}, Call{592, 24, 48, 16, true}, Call{888, 8, 130, 4, true}, Call{2000, 8, 130, 8, true}, Call{2000, 16, 16, 4, true},
             Call{74, 8, 8, 1, false}, Call{76, 64, 64, 4, false}, Call{93, 128, 64, 1, false}, Call{148, 128, 96, 1, false}, Call{148, 64, 256, 4, false}, Call{148, 64, 64, 5, false},
             Call{149, 8, 8, 1, false}, Call{149, 64, 64, 4, false}, Call{180, 64, 64, 16, false}, Call{297, 16, 16, 4, false}, Call{593, 64, 64, 16, false}, Call{888, 128, 64, 1, false},
             Call{2000, 64, 64, 16, false}, Call{2000, 64, 128, 4, false}, Call{2000, 16, 16, 32, false}, Call{2000, 128, 128, 1, false}})
        if (flow_pads_too_much(c.N, c.d, c.h, c.C) != c.off && bad++ < 9) std::printf("N=%d d=%d h=%d C=%d\n", c.N, c.d, c.h, c.C);
    return bad != 0;
}
"""


def test_many_small_sequences_take_the_kernel_that_measured_the_faster(tmp_path):
    run(tmp_path, PADDING)
