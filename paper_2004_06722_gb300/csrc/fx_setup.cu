// Fixed-point tables and factors of the block fixed-point element kernels (fx.cuh).
#include <cmath>
#include <cstring>

#include "fx.cuh"

namespace ceedbp {

namespace {

// Centro-symmetric (anti = false) or centro-antisymmetric NO x NI matrix -> even-odd tables. The
// largest absolute row sum of the scaled matrix is 2^smax, or a little less where the middle sum of a
// line product (fx.cuh: MM < 2^63 for inputs of 60 bits) asks for it. Returns 2^62 over the scale.
long double eo_tables(int NO, int NI, bool anti, const std::vector<long double>& M, int smax, std::vector<int>* limbs,
                 std::vector<double>* f64) {
  const int H = NI / 2, HC = (NI + 1) / 2, R = NO / 2;
  long double big = 0.0L;
  for (int i = 0; i < NO; ++i) {
    long double s = 0.0L;
    for (int j = 0; j < NI; ++j) s += std::fabs(M[size_t(i) * NI + j]);
    big = std::max(big, s);
  }
  auto at = [&](int i, int j) { return M[size_t(i) * NI + j]; };
  double alpha = double(std::ldexp(1.0L, smax) / big * (1.0L - 1e-9L));
  for (;; alpha *= 0.99) {
    limbs->clear();
    f64->clear();
    long double row_mm = 0.0L, worst = 0.0L;
    auto put = [&](long double v) {
      const int64_t q = int64_t(std::llrint(v * alpha)), half = int64_t(1) << 30;
      const int64_t lo = ((q + half) & ((int64_t(1) << 31) - 1)) - half, hi = (q - lo) >> 31;
      limbs->push_back(int(hi));
      limbs->push_back(int(lo));
      f64->push_back(double(v));
      // |h_M l_x| + |l_M h_x| with the folded limbs |l_x| <= 2^31, |h_x| <= 2^30
      row_mm += std::ldexp((long double)std::llabs(hi), 31) + std::ldexp((long double)std::llabs(lo), 30);
    };
    auto end_row = [&]() {
      worst = std::max(worst, row_mm);
      row_mm = 0.0L;
    };
    for (int i = 0; i < R; ++i, end_row())
      for (int j = 0; j < HC; ++j) put(j < H ? 0.5L * (at(i, j) + at(i, NI - 1 - j)) : at(i, j));
    for (int i = 0; i < R; ++i, end_row())
      for (int j = 0; j < H; ++j) put(0.5L * (at(i, j) - at(i, NI - 1 - j)));
    for (int j = 0; j < (NO % 2 ? HC : 1); ++j)  // one unused entry for an even NO
      put(NO % 2 && (j < H || !anti) ? at(R, j) : 0.0L);
    end_row();
    if (worst < std::ldexp(1.0L, 63) - std::ldexp(1.0L, 33)) return std::ldexp(1.0L, 62) / alpha;
  }
}

// (ah + al) g / w3 as limbs (|result| <= 2^62); the errors of the quotient and of the product are put back.
__device__ __forceinline__ int2 fx_factor(double g, double w3, double rw3, double ah, double al) {
  const double q = g * rw3, r = __fma_rn(-q, w3, g) * rw3;
  const double v = q * ah, d = __fma_rn(q, ah, -v) + (r * ah + q * al);
  return fx_limbs(__double2ll_rn(v) + __double2ll_rn(d) + kFxHalf);
}

// One block per element: its exponent, then the limbs of alpha G with alpha = 2^(62-k) c, where c = ch + cl in
// [1, 2) and 2^ce are mantissa and exponent of the tables' scales (their chain): one unit of the element's
// result is then exactly 2^(k+ce) units of its input. NF = 6: stiffness factors
// G [e][6][q^3] -> [e][k][3][q^2] pairs of entries (00,01), (02,11), (12,22); NF = 1: mass factors.
//
// An element is on the grid while the factors that carry it are within 2^kFxSpread of its largest row sum:
// one direction's diagonal factors at all points (collocated), the larger ones of each point (Gauss, where
// interpolation spreads every value over the element), the mass factors. A flux is known to one unit of
// the largest, and a spread of 2^7 made results up to 5 times worse than FP64's on random values (2^4: equal).
// D of orders 1 and 2 takes a constant to exact zeros in FP64, so collocated FP64 loses nothing of a function of the
// weak direction of a thin element, the grid the ratio of the factors: all three directions (all_dirs) have to
// be within 2^4 there (order 1, thickness 1/100, a function of x: 2e-14 of the result against 3e-17; from order 3
// on, and with Gauss quadrature, both arithmetics lose the same).
//
// reach: a line of nodal values counts as large while it is above 2^-reach of the element's largest value (fx.cuh).
// The ratio of the factors takes from it; the budget of `reach` bits at ratios below 2 grows at low orders, whose
// row sums are small (fixed point against FP64, worst entry in units of 2^-53 (|A||u|)_i, one node 2^6
// above the others: order 1 0.7 / 0.8, 2 2.4 / 0.9, 3 2.6 / 1.9, 5 6.4 / 2.5, 7 8.4 / 5.2, 15 20 / 7.5; 2^4: order 5 and up
// within 1.1 of FP64).
constexpr int kFxSpread = 5;
__device__ __forceinline__ int fx_reach(double big, double small, int budget) {
  if (!(small * double(1 << kFxSpread) >= big)) return 0;
  int s = 0;
  frexp(big / small, &s);  // the ratio is in [2^(s-1), 2^s)
  return max(budget + 1 - s, 0);
}

template <int NF>
__global__ void fx_factors_kernel(const double* __restrict__ G, const double* __restrict__ w, int q, double ch,
                                  double cl, int ce, int colloc, int all_dirs, int budget, void* out, int* __restrict__ gexp) {
  constexpr int NR = NF == 6 ? 5 : 2;  // largest row sum; smallest of each direction and of the points' largest
  __shared__ double sw[kMaxQ], srw[kMaxQ], sred[NR][32];
  __shared__ int s_bad;
  const int64_t e = blockIdx.x;
  const int q2 = q * q, q3 = q2 * q, tid = threadIdx.x;
  const double* Ge = G + e * NF * q3;
  if (tid < q) {
    sw[tid] = w[tid];
    srw[tid] = 1.0 / w[tid];
  }
  if (tid == 0) s_bad = 0;
  __syncthreads();
  // largest row sum of |G| and smallest diagonal entries, all without the weights
  double v[NR];
  v[0] = 0.0;
#pragma unroll
  for (int c = 1; c < NR; ++c) v[c] = __longlong_as_double(0x7fefffffffffffffll);
  bool bad = false;
  for (int p = tid; p < q3; p += blockDim.x) {
    const double rw3 = srw[p % q] * srw[(p / q) % q] * srw[p / q2];
    double f[NF];
#pragma unroll
    for (int c = 0; c < NF; ++c) {
      f[c] = fabs(Ge[size_t(c) * q3 + p]) * rw3;
      bad |= !isfinite(f[c]);
    }
    if constexpr (NF == 6) {
      v[0] = fmax(v[0], fmax(f[0] + f[1] + f[2], fmax(f[1] + f[3] + f[4], f[2] + f[4] + f[5])));
      v[1] = fmin(v[1], f[0]);
      v[2] = fmin(v[2], f[3]);
      v[3] = fmin(v[3], f[5]);
      v[4] = fmin(v[4], fmax(f[0], fmax(f[3], f[5])));
    } else {
      v[0] = fmax(v[0], f[0]);
      v[1] = fmin(v[1], f[0]);
    }
  }
  if (bad) s_bad = 1;
#pragma unroll
  for (int c = 0; c < NR; ++c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double x = __shfl_xor_sync(0xffffffffu, v[c], o);
      v[c] = c == 0 ? fmax(v[c], x) : fmin(v[c], x);
    }
    if ((tid & 31) == 0) sred[c][tid >> 5] = v[c];
  }
  __syncthreads();
  for (int i = 0; i < int(blockDim.x) / 32; ++i)
#pragma unroll
    for (int c = 0; c < NR; ++c) v[c] = c == 0 ? fmax(v[c], sred[c][i]) : fmin(v[c], sred[c][i]);
  const double big = v[0];
  int reach = 0;
  if (NF == 6 && colloc) {
    if (!all_dirs || fmin(v[1], fmin(v[2], v[3])) * 16.0 >= big)
#pragma unroll
      for (int d = 0; d < 3; ++d) reach |= fx_reach(big, v[1 + d], budget) << 4 * d;
  } else {
    reach = fx_reach(big, v[NR - 1], budget);
  }
  // big chain <= 2^k: the rows of alpha G stay within 2^62
  int k = 0;
  frexp(big * ch * (1.0 + 1e-9), &k);
  // outside the grid: not finite, spread too far, or far from 1
  const bool off = s_bad || reach == 0 || !(big > 0.0) || k > 200 || k < -200;
  if (tid == 0) gexp[e] = off ? kFxNoGrid : (k + ce) * (1 << kFxReachBits) + reach;
  if (off) return;
  const double ah = scalbn(ch, 62 - k), al = scalbn(cl, 62 - k);
  for (int p = tid; p < q3; p += blockDim.x) {
    const double w3 = sw[p % q] * sw[(p / q) % q] * sw[p / q2], rw3 = srw[p % q] * srw[(p / q) % q] * srw[p / q2];
    if constexpr (NF == 6) {
      int2 l[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) l[c] = fx_factor(Ge[size_t(c) * q3 + p], w3, rw3, ah, al);
      int4* o = static_cast<int4*>(out) + e * 3 * q3 + size_t(p / q2) * 3 * q2 + p % q2;
#pragma unroll
      for (int c = 0; c < 3; ++c) o[size_t(c) * q2] = make_int4(l[2 * c].x, l[2 * c].y, l[2 * c + 1].x, l[2 * c + 1].y);
    } else {
      static_cast<int2*>(out)[e * q3 + p] = fx_factor(Ge[p], w3, rw3, ah, al);
    }
  }
}

}  // namespace

cudaError_t launch_fx_factors(const DeviceMesh& m, int kind, const double* G, void* out, int* gexp, cudaStream_t s) {
  const double* w = m.basis + 2 * size_t(m.q) * m.p1 + size_t(m.q) * m.q;
  const int threads = m.q <= 5 ? 128 : 256;
  int e = 0;
  const long double c = 2.0L * std::frexp(kind == kStiff ? m.fx->chain : m.fx->mchain, &e);  // chain = c 2^(e-1)
  const double ch = double(c), cl = double(c - ch);
  const int all_dirs = m.colloc && m.p1 <= 3, budget = m.p1 <= 4 ? 10 - m.p1 : 5;
  if (kind == kStiff)
    fx_factors_kernel<6><<<unsigned(m.nelem), threads, 0, s>>>(G, w, m.q, ch, cl, e - 1, m.colloc, all_dirs, budget, out, gexp);
  else
    fx_factors_kernel<1><<<unsigned(m.nelem), threads, 0, s>>>(G, w, m.q, ch, cl, e - 1, m.colloc, all_dirs, budget, out, gexp);
  return cudaGetLastError();
}

// Even-odd tables of D and of the weighted transposes. With W the quadrature weights: DT = W^-1 D^T W and,
// with s_i = sum_q |J_qi| w_q, JT = s^-1 J^T W, so that W (DT f) = D^T (W f) and s (JT f) = J^T (W f).
void build_fx_tables(const Basis1D& b, FxTables* t) {
  const int p = b.p1, q = b.q;
  std::vector<long double> M(size_t(q) * q), MT(size_t(q) * q);
  for (int i = 0; i < q; ++i)
    for (int j = 0; j < q; ++j) {
      M[size_t(i) * q + j] = b.Dq[size_t(i) * q + j];
      MT[size_t(i) * q + j] = (long double)b.Dq[size_t(j) * q + i] * b.w[j] / b.w[i];
    }
  std::vector<int> no_limbs;
  std::vector<double> no_f64;
  const long double d = eo_tables(q, q, true, M, 62, &t->D, &t->D64);
  // Gauss quadrature sums the three directions before the next stage: a quarter of the range each
  const long double dt = eo_tables(q, q, true, MT, b.colloc ? 62 : 60, &t->DT, &no_f64);
  for (int i = 0; i < q; ++i)
    for (int j = 0; j < q; ++j) MT[size_t(i) * q + j] = b.Dq[size_t(j) * q + i];
  eo_tables(q, q, true, MT, 62, &no_limbs, &t->DT64);
  t->w.assign(b.rho.begin(), b.rho.end());
  t->chain = d * dt;
  if (b.colloc) return;
  std::vector<long double> J(size_t(q) * p), JT(size_t(q) * p);
  for (int j = 0; j < p; ++j) {
    long double sj = 0.0L;
    for (int i = 0; i < q; ++i) sj += std::fabs((long double)b.J[size_t(i) * p + j]) * b.w[i];
    t->w[j] = double(sj);
    for (int i = 0; i < q; ++i) {
      J[size_t(i) * p + j] = b.J[size_t(i) * p + j];
      JT[size_t(j) * q + i] = (long double)b.J[size_t(i) * p + j] * b.w[i] / t->w[j];
    }
  }
  const long double js = eo_tables(q, p, false, J, 62, &t->J, &t->J64);
  const long double jt = eo_tables(p, q, false, JT, 62, &t->JT, &no_f64);
  for (int i = 0; i < q; ++i)
    for (int j = 0; j < p; ++j) JT[size_t(j) * q + i] = b.J[size_t(i) * p + j];
  eo_tables(p, q, false, JT, 62, &no_limbs, &t->JT64);
  t->mchain = js * js * js * jt * jt * jt;
  t->chain = t->mchain * d * dt;
}

}  // namespace ceedbp
