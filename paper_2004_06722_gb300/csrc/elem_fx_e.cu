// Instantiations of the fixed-point BK5/BK6 kernel (elem_fx.cuh), p1 = 15, 16.
#include "elem_fx.cuh"

namespace ceedbp {
template cudaError_t launch_elem_fx_t<15>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<15, 1>(int64_t nelem);
template int elem_fx_blocks_t<15, 3>(int64_t nelem);
template cudaError_t launch_elem_fx_t<16>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<16, 1>(int64_t nelem);
template int elem_fx_blocks_t<16, 3>(int64_t nelem);
}  // namespace ceedbp
