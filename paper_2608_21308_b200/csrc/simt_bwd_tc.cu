// Any-shape backward: the instantiations with tensor-core products (bf16 I/O, heads wider than the block-tiled kernels take).
#include "simt_bwd.cuh"

namespace e2ttt {

int simt_bwd_launch_tc(const SimtBwdArgs& a, int kind, cudaStream_t st) {
    return kind == 0 ? launch_bwd<0, true>(a, st) : launch_bwd<1, true>(a, st);
}

}  // namespace e2ttt
