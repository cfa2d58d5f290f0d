// Instantiations of the fixed-point BK1..BK4 kernel (elem_fxgl.cuh), p1 = 2, 3, 4, 5.
#include "elem_fxgl.cuh"

namespace ceedbp {
template cudaError_t launch_elem_fxgl_t<2>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template cudaError_t launch_elem_fxgl_pair_t<2>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template int elem_fxgl_blocks_any<2>(const DeviceMesh& m);
template cudaError_t launch_elem_fxgl_t<3>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template cudaError_t launch_elem_fxgl_pair_t<3>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template int elem_fxgl_blocks_any<3>(const DeviceMesh& m);
template cudaError_t launch_elem_fxgl_t<4>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template cudaError_t launch_elem_fxgl_pair_t<4>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template int elem_fxgl_blocks_any<4>(const DeviceMesh& m);
template cudaError_t launch_elem_fxgl_t<5>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template cudaError_t launch_elem_fxgl_pair_t<5>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template int elem_fxgl_blocks_any<5>(const DeviceMesh& m);
}  // namespace ceedbp
