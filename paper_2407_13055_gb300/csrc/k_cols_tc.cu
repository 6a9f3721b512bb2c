// Tensor-core column kernels (N = 2^16 and 2^12; the smallest ring has none).
#include "cols.cuh"

namespace ckks {

template void launch_cols_tc<Geo<8, 32>, false>(const DevParams&, const TcJob&, int, int2, bool, cudaStream_t);
template void launch_cols_tc<Geo<8, 32>, true>(const DevParams&, const TcJob&, int, int2, bool, cudaStream_t);
template void launch_cols_tc<Geo<8, 8>, false>(const DevParams&, const TcJob&, int, int2, bool, cudaStream_t);
template void launch_cols_tc<Geo<8, 8>, true>(const DevParams&, const TcJob&, int, int2, bool, cudaStream_t);

}  // namespace ckks
