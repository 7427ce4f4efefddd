// What the kernels of the block-tiled reverse pass share (tile_bwd.cu, tile_chain.cu).
#pragma once
#include "simt_layout.h"
#include "tile.cuh"

namespace e2ttt {
namespace tile {

constexpr uint32_t B = 2 * kHalf;  // bytes of an operand block

// One launch of each kernel covers the chunks [c0, c0 + ng) of the call
struct GroupArgs {
    SimtBwdArgs a;
    int c0, ng;
    int s0;           // slot of chunk c0
    int first, last;  // first / last group of the call
    int shares;       // parts the chain kernel leaves of the adjoints of K^W_t, K^M_t
};
// The group whose tile_rec work runs on SMs that the chain of the group before leaves idle (ng = 0: none)
struct NextGroup {
    int c0, ng, s0;
};

__device__ __forceinline__ float* slot_of(const SimtBwdArgs& a, int seq, int g) {  // g: slot
    return reinterpret_cast<float*>(a.ws) + (size_t)seq * a.lay.per_seq + a.lay.tl.slot + (size_t)g * a.lay.tl.slot_stride;
}
__device__ __forceinline__ unsigned char* bytes_of(float* p) { return reinterpret_cast<unsigned char*>(p); }

}  // namespace tile

// The chain over the chunks with T on chip (tile_chain.cu): one CTA per 128 hidden units, h <= 1024.
inline int tile_chain_ctas(const TileLayout& tl) { return (tl.hb + 1) / 2; }
inline bool tile_chain_serves(const TileLayout& tl) { return tile_chain_ctas(tl) <= kTileMaxCl; }
// the caller sets a.cl = tile_chain_ctas, shares = 4 a.cl; next: taken along on `rec_ctas` (a multiple of a.cl) further CTAs
int tile_chain_launch(const tile::GroupArgs& ga, const tile::NextGroup& next, int rec_ctas, int kind, cudaStream_t st);

}  // namespace e2ttt
