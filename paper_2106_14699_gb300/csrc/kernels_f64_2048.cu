// FP64 forward, column, pair-product and weighted-row kernels for transform size 2048.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<double, 2048>::fwd_rows(const Geom&, const PipeArgs<double>&, bool, cudaStream_t);
template cudaError_t Sized<double, 2048>::fwd_cols(const Geom&, const PipeArgs<double>&, bool, cudaStream_t);
template cudaError_t Sized<double, 2048>::pair_cols(const Geom&, const PipeArgs<double>&, cudaStream_t);
template cudaError_t Sized<double, 2048>::pair_rows_w(const Geom&, const PipeArgs<double>&, cudaStream_t);
template cudaError_t Sized<double, 2048>::rows_w_max_blocks(int*);
}
