// Instantiations of the fixed-point BK1..BK4 kernel (elem_fxgl.cuh), p1 = 16.
#include "elem_fxgl.cuh"

namespace ceedbp {
template cudaError_t launch_elem_fxgl_t<16>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template cudaError_t launch_elem_fxgl_pair_t<16>(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s);
template int elem_fxgl_blocks_any<16>(const DeviceMesh& m);
}  // namespace ceedbp
