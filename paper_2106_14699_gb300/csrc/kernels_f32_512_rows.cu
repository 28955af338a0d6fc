// FP32 row / entropy-epilogue kernels for transform size 512.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<float, 512>::pair_rows(const Geom&, const PipeArgs<float>&, cudaStream_t);
template size_t Sized<float, 512>::rows_smem(int, bool);
template cudaError_t Sized<float, 512>::rows_max_blocks(int, bool, int*);
}
