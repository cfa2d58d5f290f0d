// Instantiations of the fixed-point BK5/BK6 kernel (elem_fx.cuh), p1 = 2, 3, 4, 5, 6.
#include "elem_fx.cuh"

namespace ceedbp {
template cudaError_t launch_elem_fx_t<2>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<2, 1>(int64_t nelem);
template int elem_fx_blocks_t<2, 3>(int64_t nelem);
template cudaError_t launch_elem_fx_t<3>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<3, 1>(int64_t nelem);
template int elem_fx_blocks_t<3, 3>(int64_t nelem);
template cudaError_t launch_elem_fx_t<4>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<4, 1>(int64_t nelem);
template int elem_fx_blocks_t<4, 3>(int64_t nelem);
template cudaError_t launch_elem_fx_t<5>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<5, 1>(int64_t nelem);
template int elem_fx_blocks_t<5, 3>(int64_t nelem);
template cudaError_t launch_elem_fx_t<6>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<6, 1>(int64_t nelem);
template int elem_fx_blocks_t<6, 3>(int64_t nelem);
}  // namespace ceedbp
