// Split 1d kernels for n = 2^11 (sgn_split_1d.cuh), a translation unit of its own so the
// instantiations compile in parallel.
#include "sgn_split_1d.cuh"

namespace sgn {
template cudaError_t split_pcg_launch<11>(const PcgArgs&, int, int, int, cudaStream_t);
template cudaError_t split_rhs_launch<11>(const RhsArgs&, int, int, int, cudaStream_t);
template cudaError_t split_linimp_launch<11>(const sp::LinArgs&, int, int, int, cudaStream_t);
template cudaError_t split_field_launch<11>(const sp::FieldArgs&, int, int, int, cudaStream_t);
}  // namespace sgn
