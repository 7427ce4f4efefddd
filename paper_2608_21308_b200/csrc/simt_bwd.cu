// Any-shape backward: dispatch, and the instantiations with fp32 FMAs (bf16 I/O, impl SIMT).
#include "simt_bwd.cuh"

namespace e2ttt {

int simt_bwd_launch_tc(const SimtBwdArgs& a, int kind, cudaStream_t st);

int simt_bwd_launch(const SimtBwdArgs& a, int kind, int io_dtype, void* stream) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (io_dtype == 0) return f64_bwd_launch(a, kind, stream);
    if (a.tc) return simt_bwd_launch_tc(a, kind, st);
    return kind == 0 ? launch_bwd<0, false>(a, st) : launch_bwd<1, false>(a, st);
}

}  // namespace e2ttt
