// FP32 row / entropy-epilogue kernels for transform size 1024.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<float, 1024>::pair_rows(const Geom&, const PipeArgs<float>&, cudaStream_t);
template size_t Sized<float, 1024>::rows_smem(int, bool);
template cudaError_t Sized<float, 1024>::rows_max_blocks(int, bool, int*);
}
