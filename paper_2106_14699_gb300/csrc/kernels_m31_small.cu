// Exact (mod 2^31 - 1) forward, column and pair-product kernels for transform sizes 16, 32, 64, 128, 256.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<m31, 16>::fwd_rows(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 16>::fwd_cols(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 16>::pair_cols(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template cudaError_t Sized<m31, 32>::fwd_rows(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 32>::fwd_cols(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 32>::pair_cols(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template cudaError_t Sized<m31, 64>::fwd_rows(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 64>::fwd_cols(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 64>::pair_cols(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template cudaError_t Sized<m31, 128>::fwd_rows(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 128>::fwd_cols(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 128>::pair_cols(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template cudaError_t Sized<m31, 256>::fwd_rows(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 256>::fwd_cols(const Geom&, const PipeArgs<m31>&, bool, cudaStream_t);
template cudaError_t Sized<m31, 256>::pair_cols(const Geom&, const PipeArgs<m31>&, cudaStream_t);
}
