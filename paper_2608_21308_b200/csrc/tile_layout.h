// Workspace of the block-tiled any-shape kernels (tile_fwd.cu, tile_bwd.cu): bf16 I/O, d <= 128, any h and C.
//
// Every matrix-product operand lives in global memory as 64 x 64 blocks of two bf16 numbers per value (hi = bf16(x),
// lo = bf16(x - hi)): 8 KB of hi, then 8 KB of lo, each 64 rows of 128 bytes with the 16-byte pieces swizzled as the MMA
// descriptors want them, so a block reaches shared memory with two bulk copies and no thread touches it.  Offsets are in
// floats, relative to the sequence's own slice of the workspace.
#pragma once
#include <stddef.h>

namespace e2ttt {

constexpr size_t kTileBlk = 4096;  // floats per block (hi + lo)
constexpr int kTileMaxD = 128;
constexpr int kTileMaxCl = 8;
constexpr int kTileShares = 4 * kTileMaxCl;

struct TileLayout {
    int db, hb, tb;  // 64-blocks along d, h and the tokens of a chunk
    int G;           // chunks the reverse pass prepares at a time
    int sets;        // sets of G slots: 2 where the chain's launch takes the next group's independent part along
    int spare;       // CTAs it has for that
    int cl;          // most CTAs per sequence
    // reverse pass, kept from launch to launch: operand blocks of the adjoints T, S of the chunk-end state
    size_t Tb[3], Sb[3];
    // forward: operand blocks of W; tokens of two chunks; intermediates of one chunk.  tile_flow.cu keeps the last matrix' blocks of odd chunks at fPzW[0]
    // (and on into fPzM[0]: 2 hb tb blocks, db hb needed), scalar kernels of two chunks at fslot, its counters at fred
    size_t Wb[3], fK[2], fQ[2], fA, fAq, fc1, fc2, fslot, fPu, fPuW, fPuM, fPzW[2], fPzM[2], fred;
    // reverse pass, intermediates of one chunk
    size_t bPhb, bZk[2], bUk, bakb, bz0[2], bslot, bdk[2], bEb[2], bred;
    // reverse pass: G slots of what does not depend on T and S (offsets inside a slot)
    size_t slot, slot_stride;
    size_t sK, sQ, sW[3], sAk, sAq, sZq[2], sPz[2], sPu, sUq, sph, sc1, sc2, sg1, sc4, sc1q, sc2q, sU, sy, spu, sr, smey, ssc, skwb, sdots;
};

// CTAs per sequence for N sequences: as many as keep every cluster resident at one CTA per SM (the driver's occupancy calculator:
// GPU processing clusters do not divide evenly into larger clusters), at most one per 64 hidden units
inline int tile_clusters_fit(int cl) {  // clusters of 1..8 CTAs that fit the GPU together
    static const int fit[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
    return fit[cl];
}
inline int tile_cluster_size(int N, int hb) {
    int cl = 1;
    for (int c = 2; c <= kTileMaxCl; ++c)
        if (N <= tile_clusters_fit(c)) cl = c;
    if (cl > hb) cl = hb;
    const int sb = (hb + cl - 1) / cl;  // hidden blocks per CTA; drop CTAs that would have none
    return (hb + sb - 1) / sb;
}

// Chunks prepared at a time: N * tb * G independent work items should fill whole waves of `ctas` CTAs, and each group costs a launch of
// every kernel.  At most 9 items per sequence, and 512 MB per set of slots for the whole call unless one slot per sequence takes more (a
// slot costs about 30 bytes per token and hidden unit): the workspace of a checkpointed call is to stay a small part of what all chunks'
// states would take.
inline int tile_group_chunks(int N, int tb, int ctas, size_t slot_bytes) {
    int best = 1;
    double best_eff = 0.0;
    for (int g = 1; g <= 9; ++g) {
        if (g > 1 && ((size_t)g * tb > 9 || slot_bytes * g * N > ((size_t)512 << 20))) break;
        const double items = (double)N * tb * g, waves = (double)(long long)((items + ctas - 1) / ctas);
        const double eff = items / (ctas * waves);
        if (eff > best_eff - 0.01) {
            best = g;
            if (eff > best_eff) best_eff = eff;
        }
    }
    return best;
}

// Appends the region behind offset o (floats); returns the end.  `chunks`: the most that one reverse launch sequence covers (those of a
// checkpointed segment, or of the call); no slot is laid out beyond them.
inline size_t tile_layout(TileLayout& t, size_t o, int N, int d, int h, int C, int nmat, bool backward, int chunks) {
    auto blocks = [](int n) { return (n + 63) / 64; };
    auto take = [&](size_t n) { size_t r = o; o += (n + 31) / 32 * 32; return r; };
    t.db = blocks(d); t.hb = blocks(h); t.tb = blocks(C);
    t.cl = tile_cluster_size(N, t.hb);
    const size_t db = t.db, hb = t.hb, tb = t.tb;
    const int sw = nmat == 3;
    const bool chain = (t.hb + 1) / 2 <= kTileMaxCl;  // tile_chain.h: S blocks of even and of odd chunks
    if (backward)
        for (int i = 0; i < nmat; ++i) { t.Tb[i] = take(db * hb * kTileBlk); t.Sb[i] = take((chain ? 2 : 1) * db * hb * kTileBlk); }
    const size_t begin = o;
    for (int i = 0; i < nmat; ++i) t.Wb[i] = take(db * hb * kTileBlk);
    for (int i = 0; i < 2; ++i) { t.fK[i] = take(tb * db * kTileBlk / 2); t.fQ[i] = take(tb * db * kTileBlk / 2); }
    t.fA = take(hb * tb * kTileBlk); t.fAq = take(hb * tb * kTileBlk);
    t.fc1 = take(hb * tb * kTileBlk); t.fc2 = take(sw * hb * tb * kTileBlk);
    t.fslot = take((size_t)t.cl * tb * 128 * db * 64);
    t.fPu = take(tb * db * kTileBlk); t.fPuW = take(tb * db * kTileBlk); t.fPuM = take(tb * db * kTileBlk);
    for (int i = 0; i < nmat - 1; ++i) { t.fPzW[i] = take(hb * tb * kTileBlk); t.fPzM[i] = take(hb * tb * kTileBlk); }
    t.fred = take((size_t)kTileMaxCl * 128);
    const size_t end_fwd = o;
    if (!backward) return end_fwd;
    o = begin;
    t.bPhb = take(hb * tb * kTileBlk);
    for (int i = 0; i < nmat - 1; ++i) { t.bZk[i] = take(hb * tb * kTileBlk); t.bz0[i] = take(hb * tb * kTileBlk); }
    t.bUk = take(tb * db * kTileBlk); t.bakb = take(hb * tb * kTileBlk);
    const int ctas = (t.hb + 1) / 2;  // of the chain kernel, where it serves
    const size_t parts = 2 * (size_t)(ctas <= kTileMaxCl && ctas > t.cl ? ctas : t.cl);
    t.bslot = take(parts * tb * 64 * db * 64);
    for (int i = 0; i < 2; ++i) {
        t.bdk[i] = take(parts * tb * 64 * db * 64);
        t.bEb[i] = take(tb * 64 * db * 64);
    }
    t.bred = take((size_t)kTileMaxCl * 128);
    t.slot = o;
    o = 0;
    t.sK = take(tb * db * kTileBlk / 2); t.sQ = take(tb * db * kTileBlk / 2);
    for (int i = 0; i < nmat; ++i) t.sW[i] = take(db * hb * kTileBlk);
    t.sAk = take(hb * tb * kTileBlk); t.sAq = take(hb * tb * kTileBlk);
    for (int i = 0; i < nmat - 1; ++i) { t.sZq[i] = take(hb * tb * kTileBlk); t.sPz[i] = take(hb * tb * kTileBlk); }
    t.sPu = take(tb * db * kTileBlk); t.sUq = take(tb * db * kTileBlk);
    t.sph = take(hb * tb * kTileBlk); t.sc1 = take(hb * tb * kTileBlk); t.sc4 = take(hb * tb * kTileBlk); t.sc1q = take(hb * tb * kTileBlk);
    t.sc2 = take(sw * hb * tb * kTileBlk); t.sg1 = take(sw * hb * tb * kTileBlk); t.sc2q = take(sw * hb * tb * kTileBlk);
    t.sU = take(tb * 128 * db * 64);
    t.sy = take(tb * 64 * db * 64); t.spu = take(tb * 64 * db * 64);
    t.sr = take(tb * 64); t.smey = take(tb * 64);
    t.ssc = take(5 * 512 + 16);
    t.skwb = take((size_t)2 * kTileShares * tb * 64);
    t.sdots = take((size_t)4 * kTileMaxCl);
    t.slot_stride = o;
    // The chain takes a CTA per 128 hidden units and sequence.  A chunk costs it about as much time as an item of the independent part:
    // with as many CTAs to spare as sequences that part is done when the chain is (chunks of one block; longer ones alike)
    t.spare = chain && ctas <= kTileMaxCl ? (tile_clusters_fit(ctas) - N) * ctas : 0;
    t.sets = t.spare >= N && o * sizeof(float) * N <= ((size_t)512 << 20) ? 2 : 1;
    t.G = tile_group_chunks(N, t.tb, t.sets == 2 ? t.spare : 148, o * sizeof(float));
    if (chunks <= t.G) {  // one group: no next one to prepare beside it
        t.G = chunks;
        t.sets = 1;
    }
    o = t.slot + t.slot_stride * (size_t)(t.sets * t.G);
    return o > end_fwd ? o : end_fwd;
}

}  // namespace e2ttt
