// Workspace layout of the any-shape kernels (host and device).  Offsets are in elements of the kernels' internal type (double for fp32 I/O:
// the fp64 kernels; float for bf16 I/O: the SIMT and the block-tiled ones), relative to the sequence's own slice.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include "tile_layout.h"

namespace e2ttt {

// ---- fp64 kernels (f64_fwd.cu, f64_bwd.cu; fp32 I/O) -----------------------------------------------------------------------
// A [tokens x d] result of a contraction over hidden units has few tiles and is cut along k; the parts are added by whoever reads it.
// From 32 tiles of 16 x 16 on there is work enough for a cluster without.  Forward and reverse pass, ms: 16 chunks of 16 tokens, d = 64,
// h = 256, one sequence 0.95, in two parts 1.00, uncut 1.16 - but 16 sequences of 64 such chunks 13.6, 13.0, 13.8.  The line at 16 tiles:
// one sequence of 512 tokens, C = 64, 0.93 -> 0.88, all else equal; at 64: 32 SwiGLU sequences of 512, d = 128, h = 384, 13.5 -> 14.7.
constexpr int kF64Parts = 4;
#ifdef __CUDACC__
#define E2TTT_HD __host__ __device__
#else
#define E2TTT_HD
#endif
E2TTT_HD inline int f64_tiles(int M, int N, int T) { return ((M + T - 1) / T) * ((N + T - 1) / T); }
// 32 x 32 tiles (half the loads per product) where a cluster of 16 has one for every CTA, else 16 x 16.  From 128 tiles on: 16 chunks of
// 16 tokens, d = 64, h = 256, one sequence 0.95 -> 1.23 ms.  From 32 on: one token of one sequence, d = 128, h = 512, 78 -> 94 us, but the
// reverse pass of 32 SwiGLU sequences of 512 tokens, h = 384, 10.1 -> 8.1 ms.
E2TTT_HD inline int f64_wide(int M, int N) { return M > 16 && N > 16 && f64_tiles(M, N, 16) >= 64; }
E2TTT_HD inline int f64_parts(int C, int d, int h) {
    const int n = (h + 63) / 64;
    return f64_tiles(C, d, 16) >= 32 ? 1 : n < kF64Parts ? n : kF64Parts;
}
// Shared memory of the forward: staging (F64Smem, f64_common.cuh), the table of jobs, scalar kernels of two chunks.  More sequences than SMs
// are bound by the latency of their phases: two CTAs share an SM, with no more than the shape needs (512 sequences of 64 tokens, d = h = 16,
// C = 1: 3658 -> 2577 us; 300 of one token, d = 64, h = 256: 898 -> 680).  An SM for each is faster with all of its registers: 64 sequences
// of 256 tokens, d = 128, h = 512 3.48 ms, on kernels with half of them 3.90.
constexpr size_t kF64FwdTile = 137216, kF64FwdTable = 10 << 10;
constexpr size_t f64_small_tile(bool wide) { return wide ? 88080 : 69648; }
constexpr size_t f64_fwd_scalars(int C) { return 16 * (size_t)(5 * C + 8); }
inline size_t f64_fwd_small(int d, int h, int C) {  // of one of two CTAs
    return f64_small_tile(f64_wide(h, d) || f64_wide(h, C) || f64_wide(d, C)) + kF64FwdTable + f64_fwd_scalars(C);
}
// (an SM has 228 KB, of which 1 KB per CTA is the system's)
inline bool f64_fwd_two(int N, int d, int h, int C) { return N > 148 && f64_fwd_small(d, h, C) <= (114 - 1) << 10; }
// Chunks that the reverse pass prepares side by side (slots): at most 64 MB of them, or one per sequence; fewer sequences than SMs take no
// more than one for every SM, or 32 MB of small ones.  ms / MB of workspace: 4096 tokens in chunks of 16, d = 64, h = 256, one sequence: 18
// chunks 9.2 / 138, 74 8.4 / 159, 148 8.7 / 187, 163 (64 MB) 8.9 / 195; 64 sequences, d = h = 16, C = 1: 3 chunks 10.2 / 137, 4 MB 7.8 / 140,
// 32 MB 7.3 / 168, 64 MB 7.5 / 200; one sequence, C = 512, d = 128, h = 512: one chunk 8.9 / 43, three of four (62 MB) 6.5 / 84; 4 SwiGLU
// sequences, d = 72, h = 200, C = 64: 16 MB 1.53 / 49, 32 MB 1.47 / 64, 64 MB 1.22 / 95.
constexpr int kF64SlotItems = 148;
constexpr size_t kF64SlotFree = (size_t)32 << 20, kF64SlotBytes = (size_t)64 << 20;
inline int f64_slots(int N, size_t slot_bytes, int chunks) {
    const size_t all = slot_bytes * (size_t)N;
    size_t g = kF64SlotBytes / all;
    if (N < kF64SlotItems) {
        const size_t each = (size_t)(kF64SlotItems + N - 1) / N, some = kF64SlotFree / all;
        g = g < (each > some ? each : some) ? g : each > some ? each : some;
    }
    return g < 1 ? 1 : g < (size_t)chunks ? (int)g : chunks;
}

// Where a chunk's tokens outweigh what the network makes of them (heads wider than their hidden units) a forward without saved states
// keeps them in three [tokens x d] places instead of seven, at two short phases more per chunk, so that no call needs more than its state,
// 3 [tokens x d], 8 [tokens x h] and 1 MiB (simt_layout).  365 tokens, d = 832, h = 1: 7.0 MiB
// instead of 16.3, 319 us instead of 317; 730 tokens 630 instead of 617.
inline bool f64_compact(int d, int h, int C, int nmat) { return (size_t)C * d > 32000 + (size_t)C * h / (size_t)(nmat - 1); }

struct F64Layout {
    int compact;
    int G;  // chunks that the reverse pass prepares at a time (slots)
    // forward: one chunk
    size_t fK[2], fQ, fA, fAq, fc1, fc2, fUk, fUq, fPu, fPuW, fPuM, fPzW[2], fPzM[2];  // fK: the keys, by the chunk's parity
    // reverse pass, chain
    size_t phb, zb[2], X2, Y2, Pub, Kb, dk, Eb, Ukb, nUkb, kwp;
    // reverse pass, slots: offsets inside a slot
    size_t slot, slot_stride;
    size_t sK, sQ, sAk, sAq, sc1, sc2, se1, se2, szq[2], sPz[2], sPzW[2], sPzM[2], sUk, sUq, sY, sPu, sPuW, sPuM, sUqb, sr, smey, ssc, skwb, sdots;
};

inline size_t f64_layout(F64Layout& f, size_t o, int N, int d, int h, int C, int nmat, bool backward, int chunks) {
    auto take = [&](size_t n) { size_t r = o; o += (n + 31) / 32 * 32; return r; };
    const size_t Ch = (size_t)C * h, Cd = (size_t)C * d, sw = nmat == 3, parts = (size_t)f64_parts(C, d, h);
    const size_t begin = o;
    f.compact = !backward && f64_compact(d, h, C, nmat);  // (one part: from 128 tiles on)
    f.fK[0] = take(Cd); f.fK[1] = f.compact ? f.fK[0] : take(Cd); f.fQ = take(Cd);
    f.fA = take(Ch); f.fAq = take(Ch); f.fc1 = take(Ch); f.fc2 = take(sw * Ch);
    f.fUk = take(parts * Cd); f.fUq = f.compact ? f.fQ : take(parts * Cd); f.fPu = f.compact ? f.fQ : take(Cd);
    // (written element by element over what they are made of, so that a call without saved states needs little more than its state)
    f.fPuW = f.fUk;
    f.fPuM = f.compact ? f.fPu : parts > 1 ? f.fUk + Cd : take(Cd);
    f.fPzW[0] = f.fc1; f.fPzW[1] = f.fc2;
    for (int i = 0; i < nmat - 1; ++i) f.fPzM[i] = take(Ch);
    const size_t end_fwd = o;
    f.G = 0;
    if (!backward) return end_fwd;
    o = begin;
    f.phb = take(Ch); f.zb[0] = take(Ch); f.zb[1] = take(sw * Ch);
    f.X2 = take(parts * Cd); f.Y2 = take(parts * Cd); f.Pub = take(parts * Cd); f.Kb = take(parts * Cd); f.dk = take(parts * Cd);
    f.Eb = take(Cd); f.Ukb = take(Cd); f.nUkb = take(Cd);
    f.kwp = take((size_t)2 * ((h + 15) / 16) * C);
    f.slot = o;
    o = 0;
    f.sK = take(Cd); f.sQ = take(Cd);
    f.sAk = take(Ch); f.sAq = take(Ch); f.sc1 = take(Ch); f.sc2 = take(sw * Ch); f.se1 = take(Ch); f.se2 = take(sw * Ch);
    for (int i = 0; i < nmat - 1; ++i) { f.szq[i] = take(Ch); f.sPz[i] = take(Ch); f.sPzW[i] = take(Ch); f.sPzM[i] = take(Ch); }
    f.sUk = take(parts * Cd); f.sUq = take(parts * Cd); f.sY = take(Cd);
    f.sPu = take(Cd); f.sPuW = take(Cd); f.sPuM = take(Cd); f.sUqb = take(Cd);
    f.sr = take(C); f.smey = take(C); f.ssc = take((size_t)2 * C + 8); f.skwb = take((size_t)2 * C);
    f.sdots = take((size_t)nmat * f64_tiles(h, d, f64_wide(h, d) ? 32 : 16) * 8 * 3);
    f.slot_stride = o;
    f.G = f64_slots(N, o * sizeof(double), chunks);
    o = f.slot + f.slot_stride * (size_t)f.G;
    return o > end_fwd ? o : end_fwd;
}

struct SimtLayout {
    // running state
    size_t W[3], M[3];
    // forward intermediates of one chunk ([2C x .] buffers hold the k-path rows first, then the q-path rows)
    size_t Z1, Z2, A, U, Pu, Pz1, Pz2;
    // backward only
    size_t T[3], S[3];   // adjoints of the chunk-end state (W, M)
    size_t Wb[3];        // adjoint accumulators of the chunk-start weights
    size_t Pa, E, XY2, XY1, Pub, Pzb, Zkb, Akb, Kb, Eb, Ukb, Uqb, Zqb;
    size_t XY1b, Pzb2, Zkb2, Zqb2;  // SwiGLU only: the second [h x d] matrix
    size_t rk, rq, red;  // per-row 1/std of the two LN calls; small reduction scratch
    size_t kWb, kMb;     // adjoints of the scalar kernels, one per token of the chunk
    size_t splitk;       // split-K partial sums of the tensor-core GEMM engine (2 * 8 * 128 * 64 elements)
    size_t rown;         // [nchunks][3][max(d,h)] row norms of the chunk-end weights before their normalisation
    size_t ckpt;         // [nchunks + 1][2][nmat][d*h] chunk-start (W, M) and, last, the final state; when states are saved.
                         // With seg > 0: [seg + 1] slots, the chunk-start states of ONE segment (recomputed by the backward)
    size_t cck;          // seg > 0: [nseg + 1][2][nmat][d*h] chunk-start states of every seg-th chunk (the checkpoints)
    int seg;             // chunks per segment (e2ttt_params.ckpt_every >= 2); 0 = the state of every chunk is kept
    size_t per_seq;      // elements per sequence
    TileLayout tl;       // region of the block-tiled kernels, when `tile`
    F64Layout fl;        // region of the fp64 kernels, when `f64`
};

// tile != 0: a call may run on the block-tiled kernels (bf16 I/O, d <= 128): their region shares the space of the SIMT
// kernels' intermediates (a call uses one of the two), behind the state that both kinds leave for each other.
// f64 != 0: fp32 I/O, which the fp64 kernels serve.  A training call has their region instead of the SIMT kernels' intermediates.  A forward
// without saved states asks for as much as those would take, twice the bytes of a bf16 call: callers of the fixed scratch (noalloc.cu)
// count by it.  The fp64 kernels' region is never larger (f64_compact).
inline SimtLayout simt_layout(int d, int h, int C, int nmat, int nchunks, bool save_states, bool backward, int seg = 0, int tile = 0, int N = 1,
                              int f64 = 0) {
    SimtLayout l{};
    size_t o = 0;
    const size_t dh = (size_t)d * h;
    auto take = [&](size_t n) { size_t r = o; o += (n + 31) / 32 * 32; return r; };
    for (int i = 0; i < 3; ++i) { l.W[i] = take(i < nmat ? dh : 0); l.M[i] = take(i < nmat ? dh : 0); }
    l.seg = save_states ? seg : 0;
    if (backward)
        for (int i = 0; i < 3; ++i) { l.T[i] = take(i < nmat ? dh : 0); l.S[i] = take(i < nmat ? dh : 0); }
    l.rown = take(save_states && l.seg == 0 ? (size_t)nchunks * 3 * (size_t)(d > h ? d : h) : 0);
    if (l.seg > 0) {
        l.ckpt = take((size_t)(l.seg + 1) * 2 * nmat * dh);
        l.cck = take((size_t)((nchunks + l.seg - 1) / l.seg + 1) * 2 * nmat * dh);
    } else {
        l.ckpt = take(save_states ? (size_t)(nchunks + 1) * 2 * nmat * dh : 0);
        l.cck = 0;
    }
    const int chunks = l.seg > 0 && l.seg < nchunks ? l.seg : nchunks;  // of a launch sequence of the reverse pass
    const size_t begin = o;
    size_t end64 = 0;
    if (f64) {
        end64 = f64_layout(l.fl, begin, N, d, h, C, nmat, backward, chunks);
        if (backward) {
            l.per_seq = end64;
            return l;
        }
    }
    l.Z1 = take((size_t)2 * C * h); l.Z2 = take((size_t)2 * C * h); l.A = take((size_t)2 * C * h);
    l.U = take((size_t)2 * C * d); l.Pu = take((size_t)C * d);
    l.Pz1 = take((size_t)C * h); l.Pz2 = take((size_t)C * h);
    if (backward) {
        for (int i = 0; i < 3; ++i) l.Wb[i] = take(i < nmat ? dh : 0);
        l.Pa = take((size_t)C * h); l.E = take((size_t)C * d);
        l.XY2 = take((size_t)C * 2 * d); l.XY1 = take((size_t)C * 2 * h);
        l.Pub = take((size_t)C * d); l.Pzb = take((size_t)C * h); l.Zkb = take((size_t)C * h);
        l.Akb = take((size_t)C * h); l.Kb = take((size_t)C * d); l.Eb = take((size_t)C * d);
        l.Ukb = take((size_t)C * d); l.Uqb = take((size_t)C * d); l.Zqb = take((size_t)C * h);
        const size_t sw = (nmat == 3) ? 1 : 0;
        l.XY1b = take(sw * C * 2 * h); l.Pzb2 = take(sw * C * h); l.Zkb2 = take(sw * C * h); l.Zqb2 = take(sw * C * h);
        l.rk = take(C); l.rq = take(C); l.red = take(64);
        l.kWb = take(C); l.kMb = take(C);
    }
    l.splitk = take((size_t)2 * 8 * 128 * 64);
    if (tile) {
        const size_t end = tile_layout(l.tl, begin, N, d, h, C, nmat, backward, chunks);
        if (end > o) o = end;
    }
    l.per_seq = end64 > o ? end64 : o;
    return l;
}

struct SimtFwdArgs {
    int N, L, d, h, C, nchunks;
    int save_states;  // 0: none; 1: the start state of every chunk -> lay.ckpt; 2: of every lay.seg-th chunk -> lay.cck
    int Ls;           // tokens between two sequences in q, k, v, o and the gates (L for a whole-sequence call; a segment
                      // call passes pointers to its first token and the full length here)
    int init_slot;    // >= 0: start from checkpoint slot init_slot of lay.cck instead of W_init / M_init; -1 otherwise
    int cl;  // CTAs per sequence (cluster size), chosen by the launcher
    int tc;  // GEMMs on the tensor cores with bf16 operands (bf16 I/O only) instead of fp32 FMAs
    int* status;  // device status word of the call (bounded waits report here)
    float eps;
    const void *q, *k, *v;
    const float *eta, *beta, *gamma;
    const float* W_init[3];
    const float* M_init[3]; // nullptr entries = zeros
    void* o;
    float* W_final[3];
    float* M_final[3];
    const float* row_norm[3];  // post-chunk normalisation targets [N, rows_i]; row_norm[0] == nullptr: none
    float norm_eps;
    void* ws;
    SimtLayout lay;
};

struct SimtBwdArgs {
    int N, L, d, h, C, nchunks;
    int Ls;           // tokens between two sequences in the token tensors (see SimtFwdArgs)
    int carry_in;     // 1: the adjoints T, S of the chunk-end state are already in the workspace (left there by the launch
                      // for the next segment); 0: read them from dW_final / dM_final
    int carry_out;    // 1: leave T, S in the workspace for the previous segment's launch; 0: write dW_init / dM_init
    int cl;  // CTAs per sequence (cluster size), chosen by the launcher
    int tc;  // GEMMs on the tensor cores with bf16 operands (bf16 I/O only) instead of fp32 FMAs
    int* status;  // device status word of the call (bounded waits report here)
    float eps;
    const void *q, *k, *v, *d_o;
    const float *eta, *beta, *gamma;
    const float* dW_final[3]; // nullptr entries = zeros
    const float* dM_final[3];
    void *dq, *dk, *dv;
    float *d_eta, *d_beta, *d_gamma;
    float* dW_init[3];
    float* dM_init[3];
    const float* row_norm[3];  // post-chunk normalisation targets [N, rows_i]; row_norm[0] == nullptr: none
    float* d_row_norm[3];      // adjoints of the targets (nullptr entries: not wanted)
    float norm_eps;
    void* ws;
    SimtLayout lay;
};

// CTAs per sequence: the largest power of two <= 8 that keeps N * cl within one wave of the GPU's SMs.  The fp64 kernels take 16 for the
// few sequences of a check (clusters above 8 are non-portable and at most 7 of 16 fit this GPU at one CTA per SM): their phases are
// chains of small products, and with 8 CTAs a CTA has several tiles of most of them.
inline int simt_cluster_size(int N, int io_dtype) {
    if (io_dtype == 0 && N <= 7) return 16;
    int cl = 1;
    while (cl < 8 && (long long)N * (cl * 2) <= 148) cl *= 2;
    return cl;
}

// What of that a device grants: `active(cl)` tells how many clusters of cl CTAs it can run at once.  Above the portable 8 that may be none
// (how the SMs are spread over processing clusters differs from board to board); every phase runs on any number of CTAs.
template <typename Q> int simt_granted_cluster(int cl, Q active) { return cl > 8 && active(cl) < 1 ? 8 : cl; }

// launchers (simt_fwd.cu / simt_bwd.cu); return a cudaError_t value as int
int simt_fwd_launch(const SimtFwdArgs& a, int kind, int io_dtype, void* stream);
int simt_bwd_launch(const SimtBwdArgs& a, int kind, int io_dtype, void* stream);
// fp32 I/O (f64_fwd.cu / f64_bwd.cu); the layout must have been made with `f64`
int f64_fwd_launch(const SimtFwdArgs& a, int kind, void* stream);
int f64_bwd_launch(const SimtBwdArgs& a, int kind, void* stream);
// the same calls on the block-tiled kernels (tile_fwd.cu / tile_bwd.cu); the layout must have been made with `tile`
int tile_fwd_launch(const SimtFwdArgs& a, int kind, void* stream);
int tile_flow_launch(const SimtFwdArgs& a, int kind, void* stream);
int tile_bwd_launch(const SimtBwdArgs& a, int kind, void* stream);

}  // namespace e2ttt
