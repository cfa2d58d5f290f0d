// Fused Jacobi-PCG kernels with device-resident scalars (Sec. 3: diagonally
// preconditioned CG around the bake-off kernels).
//
// One iteration = three launches:
//   elem   : w_L = A_L Q p and pAp = sum_e (p^e, w^e) (Algorithm 1 computes this
//            dot before the direct-stiffness sum: it needs no multiplicity
//            weighting); the last block forms alpha = rz / pAp.
//   update : w = Q^T w_L (deterministic gather-scatter, masked), then
//            r -= alpha w, z = dinv r, and the sums (r, z), (r, r);
//            the last block forms beta = rz_new / rz and tests ||r|| <= tol ||b||.
//   dir    : x += alpha p, p = dinv r + beta p (p is read once for both).
// Independent components (BP6) carry their own scalars and stop separately.
#include "gather.cuh"

namespace ceedbp {

namespace {

template <int NC>
__global__ void pcg_init_kernel(const int* __restrict__ off, const double* __restrict__ b,
                                const double* __restrict__ ax, double* __restrict__ x, double* __restrict__ r,
                                double* __restrict__ p,
                                const double* __restrict__ dinv, int64_t n, double* partials, SolveState* st,
                                double tol, int fixed) {
  __shared__ double red[256 * 3 * NC];
  double acc[3 * NC];
#pragma unroll
  for (int k = 0; k < 3 * NC; ++k) acc[k] = 0.0;
  for (int64_t g = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; g < n; g += int64_t(gridDim.x) * blockDim.x) {
    const bool dir = __ldg(off + g) < 0;
    const double di = dinv[g];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const double bv = dir ? 0.0 : b[g * NC + c];
      const double rv = dir ? 0.0 : bv - (ax ? ax[g * NC + c] : 0.0);
      const double zv = di * rv;
      if (dir) x[g * NC + c] = 0.0;
      r[g * NC + c] = rv;
      p[g * NC + c] = zv;
      acc[c] += rv * zv;
      acc[NC + c] += rv * rv;
      acc[2 * NC + c] += bv * bv;
    }
  }
  if (grid_sum_last_256<3 * NC>(acc, partials, &st->ticket[kTicketInit], red)) {
    if (threadIdx.x == 0) {
      int any = 0;
      st->ncomp = NC;
      st->fixed = fixed;
      st->x = x;
      st->step = -1;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        CompScalars& cs = st->c[c];
        cs.rz = acc[c];
        cs.rr = acc[NC + c];
        cs.bb = acc[2 * NC + c];
        cs.tol2 = tol * tol * cs.bb;
        cs.pAp = 0.0;
        cs.alpha = cs.beta = 0.0;
        cs.iters = 0;
        cs.status = isfinite(cs.rz) && isfinite(cs.rr) && isfinite(cs.bb) ? CEEDBP_OK : CEEDBP_EBREAKDOWN;
        cs.active = cs.status != CEEDBP_OK ? 0 : (fixed ? 1 : (cs.rr > cs.tol2 ? 1 : 0));
        any |= cs.active;
      }
      for (int c = NC; c < 3; ++c) st->c[c].active = 0;
      st->stop = any ? 0 : 1;
    }
  }
}

template <int NC, int U>
__global__ void __launch_bounds__(256) pcg_update_kernel(const int* __restrict__ head, const int* __restrict__ slots,
                                                         const double* __restrict__ wl, double* __restrict__ r,
                                                         const double* __restrict__ dinv, int64_t n,
                                                         double* partials, SolveState* st, int step) {
  __shared__ double red[256 * 2 * NC];
  if (st->stop) {
    if (blockIdx.x == 0 && threadIdx.x == 0) st->step = -1;  // nothing for this iteration's direction kernel
    return;
  }
  double alpha[NC];
  bool act[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    act[c] = st->c[c].active != 0;
    alpha[c] = st->c[c].alpha;
  }
  double acc[2 * NC];
#pragma unroll
  for (int k = 0; k < 2 * NC; ++k) acc[k] = 0.0;
  const int64_t stride = int64_t(gridDim.x) * 256;
  for (int64_t g0 = int64_t(blockIdx.x) * 256 + threadIdx.x; g0 < n; g0 += U * stride) {
    int hd[U];
    double w[U][NC], rv[U][NC], di[U];
#pragma unroll
    for (int h = 0; h < U; ++h) {
      const int64_t g = g0 + h * stride < n ? g0 + h * stride : g0;
      di[h] = dinv[g];
#pragma unroll
      for (int c = 0; c < NC; ++c) rv[h][c] = r[size_t(g) * NC + c];
    }
    gather_nodes<U, NC>(head, slots, wl, g0, stride, n, hd, w);
#pragma unroll
    for (int h = 0; h < U; ++h) {
      if (hd[h] == kHeadDirichlet) continue;  // Dirichlet node: x, r, p stay zero
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (!act[c]) continue;
        const double v = rv[h][c] - alpha[c] * w[h][c];
        r[size_t(g0 + h * stride) * NC + c] = v;
        acc[c] += v * (di[h] * v);
        acc[NC + c] += v * v;
      }
    }
  }
  if (grid_sum_last_256<2 * NC>(acc, partials, &st->ticket[kTicketUpdate], red)) {
    if (threadIdx.x == 0) {
      int any = 0;
      st->step = step;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        CompScalars& cs = st->c[c];
        cs.xstep = cs.active;
        if (!cs.active) continue;
        const double rz_new = acc[c];
        cs.beta = cs.rz != 0.0 ? rz_new / cs.rz : 0.0;
        cs.rz = rz_new;
        cs.rr = acc[NC + c];
        cs.iters += 1;
        if (!isfinite(rz_new)) {
          cs.status = CEEDBP_EBREAKDOWN;
          if (!st->fixed) cs.active = 0;
        }
        if (!st->fixed && cs.rr <= cs.tol2) cs.active = 0;
        any |= cs.active;
      }
      if (!any) st->stop = 1;
    }
  }
}

template <int NC>
__global__ void pcg_dir_kernel(const int* __restrict__ head, const double* __restrict__ r, double* __restrict__ p,
                               const double* __restrict__ dinv, int64_t n, const SolveState* st, int step) {
  if (st->step != step) return;  // no update ran in this iteration (the solve had stopped)
  double* __restrict__ x = st->x;
  double alpha[NC], beta[NC];
  bool xs[NC], act[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    xs[c] = st->c[c].xstep != 0;
    act[c] = st->c[c].active != 0;
    alpha[c] = st->c[c].alpha;
    beta[c] = st->c[c].beta;
  }
  for (int64_t g = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; g < n; g += int64_t(gridDim.x) * blockDim.x) {
    if (__ldg(head + g) == kHeadDirichlet) continue;
    const double di = dinv[g];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (!xs[c]) continue;
      const size_t i = size_t(g) * NC + c;
      const double pv = p[i];
      x[i] += alpha[c] * pv;
      if (act[c]) p[i] = di * r[i] + beta[c] * pv;
    }
  }
}

}  // namespace

cudaError_t launch_pcg_init(const DeviceMesh& m, const double* b, const double* ax, double* x, double* r, double* p,
                            const double* dinv, double* partials, SolveState* st, double tol, int fixed,
                            cudaStream_t s) {
  const int nb = vec_blocks(m.nglobal);
  if (m.ncomp == 3)
    pcg_init_kernel<3><<<nb, 256, 0, s>>>(m.off, b, ax, x, r, p, dinv, m.nglobal, partials, st, tol, fixed);
  else
    pcg_init_kernel<1><<<nb, 256, 0, s>>>(m.off, b, ax, x, r, p, dinv, m.nglobal, partials, st, tol, fixed);
  return cudaGetLastError();
}

cudaError_t launch_pcg_update(const DeviceMesh& m, const double* wl, double* r, const double* dinv, double* partials,
                              SolveState* st, int step, cudaStream_t s) {
  const int nb = vec_blocks(m.nglobal);
  if (m.ncomp == 3)
    pcg_update_kernel<3, 1><<<nb, 256, 0, s>>>(m.head, m.slots, wl, r, dinv, m.nglobal, partials, st, step);
  else if (gather_one(m.nglobal, nb))
    pcg_update_kernel<1, 1><<<nb, 256, 0, s>>>(m.head, m.slots, wl, r, dinv, m.nglobal, partials, st, step);
  else
    pcg_update_kernel<1, 2><<<nb, 256, 0, s>>>(m.head, m.slots, wl, r, dinv, m.nglobal, partials, st, step);
  return cudaGetLastError();
}

cudaError_t launch_pcg_dir(const DeviceMesh& m, const double* r, double* p, const double* dinv,
                           const SolveState* st, int step, cudaStream_t s) {
  const int nb = vec_blocks(m.nglobal);
  if (m.ncomp == 3)
    pcg_dir_kernel<3><<<nb, 256, 0, s>>>(m.head, r, p, dinv, m.nglobal, st, step);
  else
    pcg_dir_kernel<1><<<nb, 256, 0, s>>>(m.head, r, p, dinv, m.nglobal, st, step);
  return cudaGetLastError();
}

}  // namespace ceedbp
