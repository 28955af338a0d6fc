// FP64 forward, column, pair-product and weighted-row kernels for transform size 1024.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<double, 1024>::fwd_rows(const Geom&, const PipeArgs<double>&, bool, cudaStream_t);
template cudaError_t Sized<double, 1024>::fwd_cols(const Geom&, const PipeArgs<double>&, bool, cudaStream_t);
template cudaError_t Sized<double, 1024>::pair_cols(const Geom&, const PipeArgs<double>&, cudaStream_t);
template cudaError_t Sized<double, 1024>::pair_rows_w(const Geom&, const PipeArgs<double>&, cudaStream_t);
template cudaError_t Sized<double, 1024>::rows_w_max_blocks(int*);
}
