// 3D instantiations of the characteristic-tracing kernel family.
#include "trace_impl.cuh"

cudaError_t launch_trace_3d(TimeMode tm, int model, int mode, const TraceArgs& a, cudaStream_t s) {
    return lgnk::launch_trace_dim<3>(tm, model, mode, a, s);
}

cudaError_t launch_ell_3d(int mode, const EllArgs& a, cudaStream_t s) { return lgnk::launch_ell_dim<3>(mode, a, s); }
