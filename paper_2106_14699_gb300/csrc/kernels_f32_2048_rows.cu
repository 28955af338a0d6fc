// FP32 row / entropy-epilogue kernels for transform size 2048.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<float, 2048>::pair_rows(const Geom&, const PipeArgs<float>&, cudaStream_t);
template size_t Sized<float, 2048>::rows_smem(int, bool);
template cudaError_t Sized<float, 2048>::rows_max_blocks(int, bool, int*);
}
