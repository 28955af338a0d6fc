// FP64 forward, column, pair-product and weighted-row kernels for transform size 512.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<double, 512>::fwd_rows(const Geom&, const PipeArgs<double>&, bool, cudaStream_t);
template cudaError_t Sized<double, 512>::fwd_cols(const Geom&, const PipeArgs<double>&, bool, cudaStream_t);
template cudaError_t Sized<double, 512>::pair_cols(const Geom&, const PipeArgs<double>&, cudaStream_t);
template cudaError_t Sized<double, 512>::pair_rows_w(const Geom&, const PipeArgs<double>&, cudaStream_t);
template cudaError_t Sized<double, 512>::rows_w_max_blocks(int*);
}
