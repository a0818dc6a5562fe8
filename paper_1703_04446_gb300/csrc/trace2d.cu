// 2D instantiations of the characteristic-tracing kernel family.
#include "trace_impl.cuh"

cudaError_t launch_trace_2d(TimeMode tm, int model, int mode, const TraceArgs& a, cudaStream_t s) {
    return lgnk::launch_trace_dim<2>(tm, model, mode, a, s);
}

cudaError_t launch_ell_2d(int mode, const EllArgs& a, cudaStream_t s) { return lgnk::launch_ell_dim<2>(mode, a, s); }
