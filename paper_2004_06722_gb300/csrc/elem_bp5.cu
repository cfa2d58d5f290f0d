// Column kernel (elem.cuh) of batched BP5 solves at even orders; the reason batches keep FP64
// arithmetic stands in elem_eo.cuh.
#include "elem.cuh"

namespace ceedbp {

#define CEEDBP_BP5_P1(X) X(3) X(5) X(7) X(9) X(11) X(13) X(15)

cudaError_t launch_elem_bp5(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s) {
  switch (m.p1) {
#define X(P) \
  case P: return launch_elem_b<P, P, true, kStiff, 1, true>(m, a, s);
    CEEDBP_BP5_P1(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
}

// elements per block (block tables of batched solves)
int elem_per_block_bp5(const DeviceMesh& m) {
  switch (m.p1) {
#define X(P) \
  case P: return elem_per_block<P, P, true, 1>();
    CEEDBP_BP5_P1(X)
#undef X
    default: return 0;
  }
}

}  // namespace ceedbp
