// FP32 forward, column and pair-product kernels for transform size 4096.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<float, 4096>::fwd_rows(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 4096>::fwd_cols(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 4096>::pair_cols(const Geom&, const PipeArgs<float>&, cudaStream_t);
template int Sized<float, 4096>::tm_cols(int, int);
template cudaError_t Sized<float, 4096>::tm_max_blocks(int, int*);
}
