// Instantiations of the fixed-point BK5/BK6 kernel (elem_fx.cuh), p1 = 7, 8, 9.
#include "elem_fx.cuh"

namespace ceedbp {
template cudaError_t launch_elem_fx_t<7>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<7, 1>(int64_t nelem);
template int elem_fx_blocks_t<7, 3>(int64_t nelem);
template cudaError_t launch_elem_fx_t<8>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<8, 1>(int64_t nelem);
template int elem_fx_blocks_t<8, 3>(int64_t nelem);
template cudaError_t launch_elem_fx_t<9>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<9, 1>(int64_t nelem);
template int elem_fx_blocks_t<9, 3>(int64_t nelem);
}  // namespace ceedbp
