// Dispatch of the fixed-point kernels by order: BK5/BK6 (elem_fx.cuh, instantiated in elem_fx_[a-e].cu) and
// BK1..BK4 (elem_fxgl.cuh, instantiated in elem_fxgl_[a-h].cu).
#include "elem_fx.cuh"
#include "elem_fxgl.cuh"
#include "kernel_args.h"

namespace ceedbp {

#define CEEDBP_FX_P1(X) \
  X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12) X(13) X(14) X(15) X(16)

#define X(P)                                                                                    \
  extern template cudaError_t launch_elem_fx_t<P>(const DeviceMesh&, const ElemArgs&, cudaStream_t); \
  extern template int elem_fx_blocks_t<P, 1>(int64_t);                                          \
  extern template int elem_fx_blocks_t<P, 3>(int64_t); \
  extern template cudaError_t launch_elem_fxgl_t<P>(const DeviceMesh&, int, const ElemArgs&, cudaStream_t); \
  extern template cudaError_t launch_elem_fxgl_pair_t<P>(const DeviceMesh&, int, const ElemArgs&, cudaStream_t); \
  extern template int elem_fxgl_blocks_any<P>(const DeviceMesh&);
CEEDBP_FX_P1(X)
#undef X

cudaError_t launch_elem_fx(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s) {
  switch (m.p1) {
#define X(P) \
  case P: return launch_elem_fx_t<P>(m, a, s);
    CEEDBP_FX_P1(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
}

int elem_fx_blocks(const DeviceMesh& m) {
  switch (m.p1) {
#define X(P) \
  case P: return m.ncomp == 3 ? elem_fx_blocks_t<P, 3>(m.nelem) : elem_fx_blocks_t<P, 1>(m.nelem);
    CEEDBP_FX_P1(X)
#undef X
    default: return 0;
  }
}

cudaError_t launch_elem_fxgl(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s) {
  switch (m.p1) {
#define X(P) \
  case P: return launch_elem_fxgl_t<P>(m, kind, a, s);
    CEEDBP_FX_P1(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_elem_dfgl(const DeviceMesh& m, const ElemDfArgs& d, cudaStream_t s) {
  const int kind = m.bp == 1 ? kMass : kStiff;
  ElemArgs a{};
  a.u = d.u_f64;
  a.u_df = d.u_df;
  a.wl = reinterpret_cast<double*>(d.wl);
  a.G = d.G64;
  a.partials = d.partials;
  a.state = d.state;
  a.mask_in = d.mask_in;
  a.skip_dirichlet_out = d.skip_dirichlet_out;
  switch (m.p1) {
#define X(P) \
  case P: return launch_elem_fxgl_pair_t<P>(m, kind, a, s);
    CEEDBP_FX_P1(X)
#undef X
    default: return cudaErrorInvalidValue;
  }
}

int elem_fxgl_blocks(const DeviceMesh& m) {
  switch (m.p1) {
#define X(P) \
  case P: return elem_fxgl_blocks_any<P>(m);
    CEEDBP_FX_P1(X)
#undef X
    default: return 0;
  }
}

}  // namespace ceedbp
