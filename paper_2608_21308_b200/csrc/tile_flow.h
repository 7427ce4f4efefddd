// The forward on work items (tile_flow.cu), host and device: which calls it serves, what its items are and in which order they are handed out.
#pragma once
#include "simt_layout.h"

namespace e2ttt {

// Blocks of 64 tokens that a chunk of the call has: a call may be shorter than its chunk.  `Ls`: tokens of the whole sequence, also where a launch
// covers a segment of it, so that every launch of a call takes the same kernel
inline int flow_blocks(int C, int Ls) { return ((Ls < C ? Ls : C) + 63) / 64; }

// Whether the kernel of work items serves a call of tile_fwd_launch, or a cluster per sequence.  A tokens item has all hidden units of 64 tokens, one after the
// other, so that wide networks have a longer way through it than through the eight, six or four CTAs that up to 15, 22 or 33 sequences get; several
// blocks of tokens are items side by side but a loop to a cluster, more chunks leave items of other sequences to fill the gaps with, and more CTAs
// in clusters share the way to L2.  us, on clusters -> on work items (d = 128 and the GELU network where not said):
//   one chunk of one block    8 sequences, h = 256 49 -> 48, 384 51 -> 53, 512 51 -> 56, 2048 96 -> 135; 22, d = 64, h = 448 49 -> 62; 33, h = 1024 129 -> 140;
//                             34 153 -> 143; 64 217 -> 206; SwiGLU, h = 384, 15 sequences 70 -> 62, 20 76 -> 72
//   one chunk of two, three   128 tokens, 4 sequences, h = 768 70 -> 71, 1024 68 -> 79; 24, h = 1536 181 -> 173; 28, d = 64, h = 1024 125 -> 144;
//                             192 tokens, 4 sequences, h = 1536 135 -> 105, 22 180 -> 211
//   eight chunks of one       8 sequences, h = 384 319 -> 308, 640 354 -> 383, 1024 358 -> 503; 16, h = 512 366 -> 352, 768 385 -> 451, SwiGLU 718 -> 574;
//                             20, h = 768 586 -> 490, 2048 946 -> 1011; 24, h = 1024 848 -> 636, 4096 1951 -> 1842; d = 64: 22, h = 640 336 -> 377,
//                             24, h = 768 508 -> 435
//   four chunks of two        8 sequences, h = 768 242 -> 233, 1024 237 -> 270; 16, h = 1024 403 -> 338, 4096 1055 -> 949
//   normalised                four chunks of one: 8 sequences, h = 384 1.06, 24, h = 1024 .94, 2048 934 -> 1239 (a norm item has 64 whole rows of the last matrix);
//                             one chunk, 192 of 512 tokens, 15 sequences, h = 1024 152 -> 184
// Chunks of 512, h = 512, 64 sequences of 2048 tokens 1521 -> 1000
inline bool tile_flow_serves(const TileLayout& t, int N, int C, int Ls, int nmat, bool normed) {
    const int tb = flow_blocks(C, Ls);
    const bool one = Ls <= C;
    if (normed && t.hb > 16 && tb <= 3 && N <= 74) return false;
    if (t.hb <= (tb > 2 && N <= 16 ? (normed ? 5 : 8) : 6) * tb) return !((one || normed) && tb == 1 && nmat == 2 && t.hb > 4 && N <= 22);
    if (tb > 3 || (tb > 1 && !one)) return N > 15;
    if (one) return N > 33 || (N > 22 && (tb == 3 || (tb == 2 && t.db == 2)));
    return N > 22 || (N > 18 && t.db == 2 && t.hb <= 16) || (N > 15 && nmat == 3 && t.hb <= 24);
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
