// Launcher of the apply kernel (outputs of fixed fast weights, no update).
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace e2ttt {

struct ApplyArgs {
    int N, T, d, h;  // sequences, tokens per sequence, head dimension, hidden width
    int cl;          // CTAs per sequence (cluster size)
    int tb;          // tokens per pass (1 or 4): apply_token_block(T)
    int stage;       // stage the last matrix's block in shared memory with asynchronous copies (apply_can_stage)
    float eps;
    const void* q;   // [N, T, d] io dtype
    const float* W[3];
    void* o;         // [N, T, d] io dtype
    // set by the launcher of the one-token kernel: hidden units per CTA, ring geometry
    int per, nslots;
    uint32_t slot_bytes, ring_at;
};

// The one-token kernel: every warp's ring of `nslots` slots, each 8 rows of a first matrix or 8 rows x up to kDsCols columns of the last
constexpr int kDsWarps = 8, kDsRows = 8, kDsMaxSlots = 8;
constexpr int kDsCols = 256;                 // columns of the last matrix per piece, and the widest d this kernel takes
constexpr int kDsMaxHidden = 4096;
constexpr size_t kDsRingBytes = 96 * 1024;   // of all warps
constexpr size_t kDsFixedBytes = 9856;       // barriers and partial sums (DsShared)
struct StreamGeometry {
    int cl, per, nslots;  // CTAs per sequence, hidden units per CTA, slots per warp
    uint32_t slot_bytes, ring_at;
    size_t smem;
};
inline StreamGeometry apply_stream_geometry(int N, int d, int h) {
    StreamGeometry g{};
    // as many CTAs per sequence as keep every cluster resident at two CTAs per SM (the occupancy calculator's numbers: GPU processing
    // clusters do not divide evenly into larger clusters)
    static const int fit[9] = {0, 296, 148, 93, 71, 56, 45, 37, 33};
    g.cl = 1;
    for (int c = 2; c <= 8; ++c)
        if (N <= fit[c]) g.cl = c;
    g.per = ((h + g.cl - 1) / g.cl + 3) & ~3;
    const int cols = g.per < kDsCols ? g.per : kDsCols;
    g.slot_bytes = (uint32_t)(kDsRows * 4 * (d > cols ? d : cols));
    const int fit_slots = (int)(kDsRingBytes / (kDsWarps * g.slot_bytes));
    g.nslots = fit_slots < 1 ? 1 : fit_slots > kDsMaxSlots ? kDsMaxSlots : fit_slots;
    g.ring_at = (uint32_t)((kDsFixedBytes + (size_t)g.per * 4 + 127) / 128 * 128);
    g.smem = g.ring_at + (size_t)kDsWarps * g.nslots * g.slot_bytes;
    return g;
}
// the most any call of that kernel takes: all hidden units in one CTA, a full ring
constexpr size_t kDsMaxSmem = (kDsFixedBytes + (size_t)kDsMaxHidden * 4 + 127) / 128 * 128 + kDsRingBytes;

int apply_token_block(int T);
// CTAs per sequence: the largest power of two <= 8 that keeps all N * cl CTAs resident at two per SM
inline int apply_cluster_size(int N) {
    int cl = 1;
    while (cl < 8 && (long long)N * (cl * 2) <= 2 * 148) cl *= 2;
    return cl;
}
size_t apply_smem_bytes(int d, int cl, int tb);  // without the 64 KB staging buffer
constexpr size_t kApMaxSmem = 200 * 1024;        // the most a call may take; larger ones are refused
int apply_can_stage(int d, int h, int cl);
int apply_launch(const ApplyArgs& a, int kind, int io_dtype, void* stream);  // returns a cudaError_t value

}  // namespace e2ttt
