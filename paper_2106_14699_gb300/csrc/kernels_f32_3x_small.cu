// FP32 forward, column and pair-product kernels for the transform sizes 192, 384, 768 (3 * 2^k).
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<float, 192>::fwd_rows(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 192>::fwd_cols(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 192>::pair_cols(const Geom&, const PipeArgs<float>&, cudaStream_t);
template int Sized<float, 192>::tm_cols(int, int);
template cudaError_t Sized<float, 192>::tm_max_blocks(int, int*);
template cudaError_t Sized<float, 384>::fwd_rows(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 384>::fwd_cols(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 384>::pair_cols(const Geom&, const PipeArgs<float>&, cudaStream_t);
template int Sized<float, 384>::tm_cols(int, int);
template cudaError_t Sized<float, 384>::tm_max_blocks(int, int*);
template cudaError_t Sized<float, 768>::fwd_rows(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 768>::fwd_cols(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 768>::pair_cols(const Geom&, const PipeArgs<float>&, cudaStream_t);
template int Sized<float, 768>::tm_cols(int, int);
template cudaError_t Sized<float, 768>::tm_max_blocks(int, int*);
}
