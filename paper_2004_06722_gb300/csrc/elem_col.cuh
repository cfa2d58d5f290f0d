// FP64 BK5 element kernel of batched solves at even orders (the column kernel): w^e = A^e u^e for
// every element, the unassembled product A_L Q u of Eq. (21).  elem_eo.cuh serves the
// odd orders and says why batches run in FP64.
//
// Stiffness, Eq. (22) with J = I: w^e = sum_{m,m'} D_m^T G_mm' D_m' u^e with the
// geometric factors G of Eq. (23) (six symmetric components per point, stored
// [E][6][p1^3]); 12 p1^4 + 15 p1^3 flops per element.
//
// Layout: one element per p1*p1 thread group, thread (i, j) owns the column of
// points (i, j, 0..p1-1); the element's tiles live in shared memory; the
// t-direction column stays in registers, its contractions in even-odd form.
// Several elements share a block when p1*p1 is small.  Block tables give each
// block elements of one problem; that problem's (Q u, w^e) is summed over its
// blocks in a fixed order by the last of them, which forms alpha.
#pragma once

#include "common.cuh"

namespace ceedbp {

// Even-odd form (Eq. (37)) of a product y = M x with M centro-symmetric
// (SIGN = +1: M[A-1-a][B-1-b] = M[a][b], the interpolation J and J^T) or
// centro-antisymmetric (SIGN = -1: the derivative D and D^T).  With
// x+_b = x_b + x_{B-1-b}, x-_b = x_b - x_{B-1-b} (b < B/2) and the half tables
// E = (M[a][b] + M[a][B-1-b]) / 2, O = (M[a][b] - M[a][B-1-b]) / 2 of the top
// rows (a < (A+1)/2), plus the middle column M[a][B/2] when B is odd:
//   y_a = S_E + S_O,  y_{A-1-a} = SIGN (S_E - S_O),
// and for odd A the middle row is S_E (SIGN = +1) or S_O (SIGN = -1).  About
// half the multiply-adds of the direct product; used for the contractions
// that stay in a thread's registers.
template <int A, int B>
struct EoTab {
  static constexpr int HA = (A + 1) / 2, HB = B / 2;
  static constexpr int SIZE = 2 * HA * HB + HA;  // [E HA x HB][O HA x HB][middle column HA]
};

// tables of row-major M (A x B, leading dimension ld, element (a, b) at M[a * ld + b],
// or M[b * ld + a] when TRANS) into T
template <int A, int B, bool TRANS>
__device__ __forceinline__ void eo_build(const double* M, int ld, double* T, int tid, int nthr) {
  using E = EoTab<A, B>;
  for (int q = tid; q < E::HA * E::HB; q += nthr) {
    const int ra = q / E::HB, cb = q % E::HB;
    const double m0 = TRANS ? M[cb * ld + ra] : M[ra * ld + cb];
    const double m1 = TRANS ? M[(B - 1 - cb) * ld + ra] : M[ra * ld + B - 1 - cb];
    T[q] = 0.5 * (m0 + m1);
    T[E::HA * E::HB + q] = 0.5 * (m0 - m1);
  }
  if constexpr (B % 2 == 1)
    for (int ra = tid; ra < E::HA; ra += nthr) T[2 * E::HA * E::HB + ra] = TRANS ? M[(B / 2) * ld + ra] : M[ra * ld + B / 2];
}

template <int A, int B, int SIGN>
__device__ __forceinline__ void eo_mul(const double* T, const double (&x)[B], double (&y)[A]) {
  using E = EoTab<A, B>;
  constexpr int HA = E::HA, HB = E::HB;
  const double* TE = T;
  const double* TO = T + HA * HB;
  const double* TM = T + 2 * HA * HB;
  double xe[HB > 0 ? HB : 1], xo[HB > 0 ? HB : 1];
#pragma unroll
  for (int b = 0; b < HB; ++b) {
    xe[b] = x[b] + x[B - 1 - b];
    xo[b] = x[b] - x[B - 1 - b];
  }
  // the odd half-sum accumulates on top of the even one: y[ra] = S_E + S_O leaves the chain and
  // the mirror output is one fma of it (one FP64 operation fewer per output pair)
#pragma unroll
  for (int ra = 0; ra < A / 2; ++ra) {
    double se = 0.0;
#pragma unroll
    for (int b = 0; b < HB; ++b) se += TE[ra * HB + b] * xe[b];
    if constexpr (B % 2 == 1) se += TM[ra] * x[B / 2];
    double s = se;
#pragma unroll
    for (int b = 0; b < HB; ++b) s = __fma_rn(TO[ra * HB + b], xo[b], s);
    y[ra] = s;                                                               // S_E + S_O
    y[A - 1 - ra] = SIGN > 0 ? __fma_rn(2.0, se, -s) : __fma_rn(-2.0, se, s);  // S_E - S_O or S_O - S_E
  }
  if constexpr (A % 2 == 1) {
    constexpr int ra = A / 2;
    double sm = 0.0;
#pragma unroll
    for (int b = 0; b < HB; ++b) sm += SIGN > 0 ? TE[ra * HB + b] * xe[b] : TO[ra * HB + b] * xo[b];
    if constexpr (SIGN > 0 && B % 2 == 1) sm += TM[ra] * x[B / 2];
    y[ra] = sm;
  }
}

template <int P1>
constexpr int elem_col_per_block() {
  return 256 / (P1 * P1) < 1 ? 1 : 256 / (P1 * P1);
}
template <int P1>
constexpr int elem_col_threads() {  // whole warps
  return (elem_col_per_block<P1>() * P1 * P1 + 31) / 32 * 32;
}

template <int P1>
__global__ void __launch_bounds__(elem_col_threads<P1>()) elem_col_kernel(const DeviceMesh m, const ElemArgs a) {
  constexpr int PP = P1 * P1, P3 = PP * P1;
  extern __shared__ double smem[];
  double* sD = smem;         // [P1][P1]
  double* red = sD + PP;     // 32
  double* tD = red + 32;     // even-odd tables of D, D^T
  double* tDT = tD + EoTab<P1, P1>::SIZE;
  double* ebuf = tDT + EoTab<P1, P1>::SIZE;

  const int tid = threadIdx.x;
  const int slot = tid / PP, t = tid - slot * PP;
  const int tx = t % P1, ty = t / P1;
  const int prob = a.blk_prob[blockIdx.x];
  if (!a.bst[prob].c.active) return;
  const int64_t e = a.blk_e0[blockIdx.x] + slot;
  const bool active = slot < a.blk_n[blockIdx.x];

  for (int i = tid; i < PP; i += blockDim.x) sD[i] = m.basis[2 * PP + i];
  // read by every thread only after the barrier that follows the gather
  eo_build<P1, P1, false>(m.basis + 2 * PP, P1, tD, tid, blockDim.x);
  eo_build<P1, P1, true>(m.basis + 2 * PP, P1, tDT, tid, blockDim.x);

  double* sU = ebuf + size_t(active ? slot : 0) * 3 * P3;
  double* sR = sU + P3;
  double* sS = sR + P3;
  const int* l2g = m.l2g + e * P3;
  double uq[P1], tq[P1], vq[P1];
  if (active) {  // gather u^e = Q u (Eq. (21)); Dirichlet nodes read as 0 when masking
#pragma unroll
    for (int z = 0; z < P1; ++z) {
      const int g = __ldg(l2g + z * PP + t);
      if (g >= 0) uq[z] = __ldg(a.u + g);
      else uq[z] = a.mask_in ? 0.0 : __ldg(a.u + (-g - 1));
      sU[z * PP + t] = uq[z];
    }
  }
  __syncthreads();
  if (active) {
    const double* G = a.G + e * 6 * P3;
    // t derivatives of the whole column first; tq[z] holds u_t until it becomes the t part of G grad u
    eo_mul<P1, P1, -1>(tD, uq, tq);
#pragma unroll
    for (int z = 0; z < P1; ++z) {
      const int pt = z * PP + t;
      const double g00 = __ldcs(G + 0 * P3 + pt), g01 = __ldcs(G + 1 * P3 + pt), g02 = __ldcs(G + 2 * P3 + pt);
      const double g11 = __ldcs(G + 3 * P3 + pt), g12 = __ldcs(G + 4 * P3 + pt), g22 = __ldcs(G + 5 * P3 + pt);
      double ur = 0.0, us = 0.0;
      const double ut = tq[z];
#pragma unroll
      for (int n = 0; n < P1; ++n) {
        ur += sD[tx * P1 + n] * sU[z * PP + ty * P1 + n];
        us += sD[ty * P1 + n] * sU[z * PP + n * P1 + tx];
      }
      sR[pt] = g00 * ur + g01 * us + g02 * ut;
      sS[pt] = g01 * ur + g11 * us + g12 * ut;
      tq[z] = g02 * ur + g12 * us + g22 * ut;
    }
  }
  __syncthreads();
  double dot[1] = {0.0};
  if (active) {
    eo_mul<P1, P1, -1>(tDT, tq, vq);
    double* wl = a.wl + size_t(e) * P3;
#pragma unroll
    for (int z = 0; z < P1; ++z) {
      double v = vq[z];
#pragma unroll
      for (int n = 0; n < P1; ++n) {
        v += sD[n * P1 + tx] * sR[z * PP + ty * P1 + n];
        v += sD[n * P1 + ty] * sS[z * PP + n * P1 + tx];
      }
      const int idx = z * PP + t;
      if (!(a.skip_dirichlet_out && __ldg(l2g + idx) < 0)) wl[idx] = v;
      dot[0] += v * uq[z];
    }
  }
  batch_alpha(dot, a.partials, a.prob_blk0, a.prob_nblk, a.bst, prob, red);
}

template <int P1>
cudaError_t launch_elem_col_t(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s) {
  const size_t smem = sizeof(double) * (size_t(P1) * P1 + 32 + 2 * EoTab<P1, P1>::SIZE +
                                        size_t(elem_col_per_block<P1>()) * 3 * P1 * P1 * P1);
  auto kern = elem_col_kernel<P1>;
  // set once per instantiation (not a stream operation; kept out of graph capture)
  static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (attr != cudaSuccess) return attr;
  kern<<<unsigned(a.batch_blocks), elem_col_threads<P1>(), smem, s>>>(m, a);
  return cudaGetLastError();
}

}  // namespace ceedbp
