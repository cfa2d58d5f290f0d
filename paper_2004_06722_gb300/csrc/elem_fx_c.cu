// Instantiations of the fixed-point BK5/BK6 kernel (elem_fx.cuh), p1 = 10, 11, 12.
#include "elem_fx.cuh"

namespace ceedbp {
template cudaError_t launch_elem_fx_t<10>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<10, 1>(int64_t nelem);
template int elem_fx_blocks_t<10, 3>(int64_t nelem);
template cudaError_t launch_elem_fx_t<11>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<11, 1>(int64_t nelem);
template int elem_fx_blocks_t<11, 3>(int64_t nelem);
template cudaError_t launch_elem_fx_t<12>(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s);
template int elem_fx_blocks_t<12, 1>(int64_t nelem);
template int elem_fx_blocks_t<12, 3>(int64_t nelem);
}  // namespace ceedbp
