// Exact (mod 2^31 - 1) row / entropy-epilogue kernels for transform sizes 16, 32, 64, 128, 256.
#include "pipeline_impl.cuh"
namespace cmif {
template cudaError_t Sized<m31, 16>::pair_rows(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template cudaError_t Sized<m31, 16>::pair_rows_counts(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template size_t Sized<m31, 16>::rows_smem(int, bool);
template cudaError_t Sized<m31, 16>::rows_max_blocks(int, bool, int*);
template cudaError_t Sized<m31, 32>::pair_rows(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template cudaError_t Sized<m31, 32>::pair_rows_counts(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template size_t Sized<m31, 32>::rows_smem(int, bool);
template cudaError_t Sized<m31, 32>::rows_max_blocks(int, bool, int*);
template cudaError_t Sized<m31, 64>::pair_rows(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template cudaError_t Sized<m31, 64>::pair_rows_counts(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template size_t Sized<m31, 64>::rows_smem(int, bool);
template cudaError_t Sized<m31, 64>::rows_max_blocks(int, bool, int*);
template cudaError_t Sized<m31, 128>::pair_rows(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template cudaError_t Sized<m31, 128>::pair_rows_counts(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template size_t Sized<m31, 128>::rows_smem(int, bool);
template cudaError_t Sized<m31, 128>::rows_max_blocks(int, bool, int*);
template cudaError_t Sized<m31, 256>::pair_rows(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template cudaError_t Sized<m31, 256>::pair_rows_counts(const Geom&, const PipeArgs<m31>&, cudaStream_t);
template size_t Sized<m31, 256>::rows_smem(int, bool);
template cudaError_t Sized<m31, 256>::rows_max_blocks(int, bool, int*);
}
