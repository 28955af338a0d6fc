// Exact (mod 2^31 - 1) forward, column and pair-product kernels for transform size 1024.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<m31, 1024>::fwd_rows(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 1024>::fwd_cols(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 1024>::pair_cols(const Geom&, const PipeArgs<m31>&, cudaStream_t);
}
