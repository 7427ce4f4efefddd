// Any-shape backward: the instantiations with fp64 arithmetic (fp32 I/O).
#include "simt_bwd.cuh"

namespace e2ttt {

int simt_bwd_launch_f64(const SimtBwdArgs& a, int kind, cudaStream_t st) {
    return kind == 0 ? launch_bwd<double, float, 0, false>(a, st) : launch_bwd<double, float, 1, false>(a, st);
}

}  // namespace e2ttt
