// Column kernel (elem_col.cuh) of batched BP5 solves at even orders.
#include "elem_col.cuh"

namespace ceedbp {

#define CEEDBP_COL_P1(X) X(3) X(5) X(7) X(9) X(11) X(13) X(15)

cudaError_t launch_elem_col(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s) {
  switch (m.p1) {
#define X(P) \
  case P: return launch_elem_col_t<P>(m, a, s);
    CEEDBP_COL_P1(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
}

// elements per block (block tables of batched solves)
int elem_col_per_block_rt(const DeviceMesh& m) {
  switch (m.p1) {
#define X(P) \
  case P: return elem_col_per_block<P>();
    CEEDBP_COL_P1(X)
#undef X
    default: return 0;
  }
}

}  // namespace ceedbp
