// FP32 Tensor-Memory row / entropy-epilogue kernel over several units (rotation
// angles) for transform sizes 1536, 3072 and 4096.
#include "pipeline_impl.cuh"
namespace cmif {
template <int Q, bool NMI>
cudaError_t launch_rows_tm_units(const Geom& g, const PipeArgs<float>& a, cudaStream_t s) {
    return launch_rows_tm_mode<Q, NMI, 1>(g, a, s);
}
template cudaError_t launch_rows_tm_units<1536, false>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<1536, true>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<3072, false>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<3072, true>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<4096, false>(const Geom&, const PipeArgs<float>&, cudaStream_t);
template cudaError_t launch_rows_tm_units<4096, true>(const Geom&, const PipeArgs<float>&, cudaStream_t);
}  // namespace cmif
