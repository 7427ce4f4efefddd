// The forward on work items (tile_flow.cu), host and device: which calls it serves, what its items are and in which order they are handed out.
#pragma once
#include "simt_layout.h"

namespace e2ttt {

// Blocks of 64 tokens that a chunk of the call has: a call may be shorter than its chunk.  `Ls`: tokens of the whole sequence, also where a launch
// covers a segment of it, so that every launch of a call takes the same kernel
inline int flow_blocks(int C, int Ls) { return ((Ls < C ? Ls : C) + 63) / 64; }

// Whether the kernel of work items serves a call of tile_fwd_launch, or a cluster per sequence.  A tokens item has all hidden units of 64 tokens, one after the
// other, so that wide networks have a longer way through it than through the eight, six or four CTAs that up to 15, 22 or 33 sequences get; several
// blocks of tokens are items side by side but a loop to a cluster, and more CTAs in clusters share the way to L2.  It does not go by the number of chunks, so that
// a sequence given in several calls of whole chunks has the same bits as in one; single chunks are the worse for work items (a queue filled and
// drained at once), and the lines lie where calls of one and of four chunks balance.  Time on work items / on clusters, one chunk, four chunks (d = 128 and
// the GELU network where not said; 7000 calls measured):
//   one block     8 sequences, h = 256 .96 .87, 384 1.06 .98, 512 1.12 1.10, 1024 1.39 1.40; d = 64, 33, h = 512 1.17 1.04; 22, h = 512 1.08 .87, 640 1.17 .86, 768 1.12 .84,
//                 1024 1.17 .96; 23, h = 512 .96 .87, 1024 1.03 .78, 2048 1.12 .96; 28, h = 2048 1.10 .85; SwiGLU: 16, h = 512 .90 .86, 768 1.07 .86, 1024 1.13 .97
//   two blocks    15 sequences, h = 768 .92 .76, 1024 1.12 .87; 16, h = 1024 .94 .81, 1536 1.05 .85, 2048 1.06 .91; 22, h = 2048 1.08 .90
//   three, four   8 sequences, h = 1536 .91 .76, 2048 1.00 .87 | .93 .80; 15, h = 2048 1.09 .87 | .99 .79; 22 1.14 .79 | .98 .72; 64, h = 512 .77 .60 | .74 .60
//   normalised    (a norm item has 64 whole rows of the last matrix)  one block: 8 sequences, h = 384 1.03 1.05, 22, h = 640 1.15 .94, 33, h = 1024 1.16 1.00, 64, h = 2048
//                 1.06 1.09; d = 64: 33, h = 512 1.06 1.12, SwiGLU 22 .89 .99; two: SwiGLU, 15, h = 640 .88 .90, 768 1.05 .88; d = 64, 22, h = 640 .98 .92, 768 1.18 1.08; four: 22, h = 2048 1.11 1.06, 23 .95 .93
// What clusters take changes from GPU to GPU, with where they fit: 16 sequences, h = 512, one block 54 and 67 us (four chunks 183, 195), on work items 57 (184); normalised,
// h = 384 1.03 and .85.  Chunks of 512, h = 512, 64 sequences of 2048 tokens 1521 -> 1000 us
inline bool tile_flow_serves(const TileLayout& t, int N, int C, int Ls, int nmat, bool normed) {
    const int tb = flow_blocks(C, Ls), hb = t.hb;
    const bool wide = t.db == 2, sw = nmat == 3;
    if (normed && hb > 16 && tb <= 3 && N <= 74) return false;
    if (tb > 2) return hb <= (normed ? 5 : 8) * tb || N > (normed && hb > 24 ? 22 : 15);
    if (tb == 2) return hb <= (wide || (normed && sw) ? 12 : normed ? 6 : 10) || N > (hb > 24 || (normed && hb > 8) ? 22 : 15);
    if (hb <= 4) return true;
    if (normed) {
        if (hb <= 6) return N > (wide ? 15 : 22) || sw;
        return N > (sw && hb <= (wide ? 12 : 8) ? 15 : hb <= 8 && wide ? 15 : hb <= 12 && (wide || sw) ? 22 : 33);
    }
    if (hb <= 6) return true;
    if (hb > 16) return N > 24;
    if (sw) return N > (hb <= (wide ? 12 : 8) ? 15 : 22);
    return N > (wide ? (hb <= 8 ? 15 : 18) : hb <= 8 ? 33 : 24);
}

// Many sequences of small states in chunks of a few tokens (GELU network, at most 1024 hidden units): a block of 64 tokens is then mostly padding, and
// simt_fwd.cu, one CTA per sequence, can be the faster.  Its time goes by waves of 148 sequences; work items go to any CTA, so that theirs goes by
// sequences, and a call fills and drains their queue once.  The sums below are us of a wave and of 148 sequences per chunk, after 5700 calls of 76 to 2000
// sequences on both kernels.  It does not go by the number of chunks, so that a sequence given in several calls has the same bits as
// in one: the line is where calls of two chunks break even.  us, there -> on work items, one chunk / four:
//   C = 1   148 sequences, d = h = 64 43 -> 69 / 144 -> 176; 8 x 600 135 -> 196 / 499 -> 560; 64 x 192 105 -> 91 / 279 -> 271; 128 x 128 119 -> 97 / 269 -> 219
//           100, d = h = 16 38 -> 53 / 128 -> 139; 64 x 72 49 -> 57 / 160 -> 148;  149, 64 x 64, two waves, 80 -> 70 / 270 -> 176;  592, 64 x 64 181 -> 190 / 588 -> 635
//   C = 16  888, d = h = 16 231 -> 258 / 830 -> 917; 64 x 64 307 -> 276 / 952 -> 948; 128 x 16 315 -> 300 / 1121 -> 993;  C = 32  888, 8 x 8 255 -> 253 / 926 -> 907
inline bool flow_pads_too_much(int N, int d, int h, int C) {
    const int dh = d * h;
    if (N <= 74 || dh > (C <= 4 ? 16384 : C <= 16 ? 12288 : C <= 32 && h <= 256 ? 9216 : 0) || (N <= 148 && C > 4)) return false;
    const float waves = (float)((N + 147) / 148), tiles = (float)((h + 127) / 128), more = d > 64 ? 1.0f : 0.0f;
    const float there = 5.0f + 23.0f * tiles + (h <= 64 ? 3.0f : h <= 128 ? 8.0f : 0.0f) + 9.0f * more + 1.2e-3f * dh + (dh > 8192 ? 1.5e-3f * (dh - 8192) : 0.0f) +
                        (C > 4 ? (0.13f + 0.06f * tiles + 2e-5f * dh) * C : 0.0f);
    const float here = 13.5f + 24.5f * tiles + 2.5f * more + 2e-4f * dh, once = 18.0f - 3.0f * waves;
    return waves * there < here * N / 148.0f + (once > 0.0f ? once : 0.0f);
}

struct FlowPlan {
    int N, L, C, nchunks;       // the launch
    int tb;                     // blocks of 64 tokens of a chunk
    int sets, gs, off2, off3;   // sets of gs sequences; a sequence's weights (norm) items come off2 (off3) steps after its tokens
    int steps, slots;           // steps of a set, items of a step
    int ns, n2, n3;             // slices of 128 hidden units; weights items, norm items of a chunk
};
inline FlowPlan flow_plan(const TileLayout& tl, int N, int L, int C, int nmat, bool normed) {
    FlowPlan f{};
    f.N = N; f.L = L; f.C = C;
    f.nchunks = (L + C - 1) / C;
    f.tb = flow_blocks(C, L);
    f.ns = (tl.hb + 1) / 2;
    f.n2 = nmat * f.ns;
    f.n3 = normed ? (nmat - 1) * f.ns + tl.db : 0;
    f.slots = f.tb + f.n2 + f.n3;
    // How long the items take (thousand cycles, measured), and with it how many sequences keep the GPU busy while each waits for its own
    // chain of items, with a third to spare; fewer sequences at a time are better for L2.  A sequence's weights and norm items are put off by as much as
    // what they depend on takes
    const double t1 = 20 + (nmat == 2 ? 11 : 14) * f.ns, t2 = 15 + 7.5 * f.tb, t2last = 15 + 3.5 * f.tb, t3 = f.n3 ? 10 : 0;
    const double chain = t1 + t2 + t3, work = f.tb * t1 + f.ns * ((nmat - 1) * t2 + t2last) + f.n3 * t3;
    const int enough = (int)(1.33 * 148 * chain / work) + 1;
    f.sets = N / enough < 1 ? 1 : N / enough;
    f.gs = (N + f.sets - 1) / f.sets;
    f.sets = (N + f.gs - 1) / f.gs;
    f.off2 = (int)(f.gs * t1 / chain);
    f.off3 = f.n3 ? (int)(f.gs * (t1 + t2) / chain) : 0;
    if (f.nchunks == 1 && N * f.tb <= 148 && N * f.slots > 148) {
        // One chunk, a CTA for every tokens item but not for every item: tokens first, or the last of them wait for CTAs that wait for the first (64 sequences
        // of 64 tokens, d = 64, h = 192 62 -> 54 us, on clusters 56; 148, h = 64 68 -> 56, 59)
        f.sets = 1;
        f.gs = f.off2 = N;
        f.off3 = f.n3 ? 2 * N : 0;
    }
    f.steps = f.nchunks * f.gs + (f.off3 > f.off2 ? f.off3 : f.off2);
    return f;
}

enum { kFlowNone, kFlowTokens, kFlowWeights, kFlowNorm, kFlowEnd };
struct FlowItem {
    int type, seq, c, part;
};
// Item `id` of the queue.  Every item comes after those that it depends on (tokens: the chunk before's weights or norms; weights: the chunk's
// tokens; norms: its weights)
E2TTT_HD inline FlowItem flow_item(const FlowPlan& f, long long id) {
    const long long per = (long long)f.steps * f.slots;
    const int set = (int)(id / per);
    if (set >= f.sets) return {kFlowEnd, 0, 0, 0};
    const long long r = id - set * per;
    const int step = (int)(r / f.slots), slot = (int)(r - (long long)step * f.slots);
    FlowItem it;
    int j = step;
    if (slot < f.tb) { it.type = kFlowTokens; it.part = slot; }
    else if (slot < f.tb + f.n2) { it.type = kFlowWeights; it.part = slot - f.tb; j -= f.off2; }
    else { it.type = kFlowNorm; it.part = slot - f.tb - f.n2; j -= f.off3; }
    if (j < 0 || j >= f.nchunks * f.gs) return {kFlowNone, 0, 0, 0};
    it.c = j / f.gs;
    it.seq = set * f.gs + j - it.c * f.gs;
    if (it.seq >= f.N || (it.type == kFlowTokens && it.part * 64 >= f.L - it.c * f.C)) it.type = kFlowNone;
    return it;
}

}  // namespace e2ttt
