// Exact (mod 2^31 - 1) forward, column and pair-product kernels for transform size 4096.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<m31, 4096>::fwd_rows(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 4096>::fwd_cols(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 4096>::pair_cols(const Geom&, const PipeArgs<m31>&, cudaStream_t);
}
