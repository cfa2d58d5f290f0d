// Even-odd FP64 BK5 kernel of batched solves, even p1 (odd orders 1..15), see elem_eo.cuh.
#include "elem_eo.cuh"

namespace ceedbp {

#define CEEDBP_EO_P1(X) X(2) X(4) X(6) X(8) X(10) X(12) X(14) X(16)

cudaError_t launch_elem_eo(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s) {
  switch (m.p1) {
#define X(P) \
  case P: return launch_elem_eo_t<P>(m, a, s);
    CEEDBP_EO_P1(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
}

int elem_eo_per_block_rt(const DeviceMesh& m) {
  switch (m.p1) {
#define X(P) \
  case P: return elem_eo_per_block<P>();
    CEEDBP_EO_P1(X)
#undef X
    default: return 0;
  }
}

}  // namespace ceedbp
