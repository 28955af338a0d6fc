// FP32 Tensor-Memory row / entropy-epilogue kernel over several units (rotation
// angles) for transform sizes 512, 1024 and 2048.
#include "pipeline_impl.cuh"
namespace cmif {
template <int Q, bool NMI>
cudaError_t launch_rows_tm_units(const Geom& g, const PipeArgs<float>& a, cudaStream_t s) {
    return launch_rows_tm_mode<Q, NMI, 1>(g, a, s);
}
template cudaError_t launch_rows_tm_units<512, false>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<512, true>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<1024, false>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<1024, true>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<2048, false>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<2048, true>(const Geom&, const PipeArgs<float>&, cudaStream_t);
}  // namespace cmif
