// FP32 forward, column and pair-product kernels for transform sizes 16, 32, 64, 128, 256.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<float, 16>::fwd_rows(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 16>::fwd_cols(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 16>::pair_cols(const Geom&, const PipeArgs<float>&, cudaStream_t);
template int Sized<float, 16>::tm_cols(int, int);
template cudaError_t Sized<float, 16>::tm_max_blocks(int, int*);
template cudaError_t Sized<float, 32>::fwd_rows(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 32>::fwd_cols(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 32>::pair_cols(const Geom&, const PipeArgs<float>&, cudaStream_t);
template int Sized<float, 32>::tm_cols(int, int);
template cudaError_t Sized<float, 32>::tm_max_blocks(int, int*);
template cudaError_t Sized<float, 64>::fwd_rows(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 64>::fwd_cols(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 64>::pair_cols(const Geom&, const PipeArgs<float>&, cudaStream_t);
template int Sized<float, 64>::tm_cols(int, int);
template cudaError_t Sized<float, 64>::tm_max_blocks(int, int*);
template cudaError_t Sized<float, 128>::fwd_rows(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 128>::fwd_cols(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 128>::pair_cols(const Geom&, const PipeArgs<float>&, cudaStream_t);
template int Sized<float, 128>::tm_cols(int, int);
template cudaError_t Sized<float, 128>::tm_max_blocks(int, int*);
template cudaError_t Sized<float, 256>::fwd_rows(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 256>::fwd_cols(const Geom&, const PipeArgs<float>&, bool, cudaStream_t);
template cudaError_t Sized<float, 256>::pair_cols(const Geom&, const PipeArgs<float>&, cudaStream_t);
template int Sized<float, 256>::tm_cols(int, int);
template cudaError_t Sized<float, 256>::tm_max_blocks(int, int*);
}
