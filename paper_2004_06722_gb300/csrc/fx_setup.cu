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

// Magnitude of a product g c / w as an upper word of FP64 would order it: 20 bits below the exponent field e,
// for (1 + fraction) 2^(e-1022); the product's upper bits cut, zeros and subnormal g zero.
__device__ __forceinline__ int fx_key(double g, FxWeight f) {
  const int hi = __double2hiint(g), ev = (hi >> 20) & 0x7ff;
  const unsigned p = __umulhi(unsigned((hi & 0xfffff) | 0x100000) << 11, unsigned(f.m >> 32));
  const int up = int(p >> 31);  // 2^30 <= p < 2^32
  return ev == 0 ? 0 : ((ev + f.x - 1 + up) << 20) | int((p >> (10 + up)) & 0xfffffu);
}

// Upper bound of a sum of three magnitudes of at most `top`'s exponent: each is cut by at most 2^-19.
__device__ __forceinline__ int fx_key_sum(int a, int b, int c, int top) {
  const int e = top >> 20;
  auto rel = [&](int k) {
    const int d = (k >> 20) - e;
    return d < -60 ? 0.0f : __int_as_float(((127 + d) << 23) | ((k & 0xfffff) << 3));
  };
  return (__float_as_int(rel(a) + rel(b) + rel(c)) >> 3) + ((e - 127) << 20) + 8;
}

// g c / w 2^(62-k) as limbs (|result| <= 2^62), to 2^-62 of itself.
__device__ __forceinline__ int2 fx_factor(double g, FxWeight f, int k) {
  const int hi = __double2hiint(g), ev = (hi >> 20) & 0x7ff;
  const unsigned long long m =
      ((unsigned long long)(unsigned((hi & 0xfffff) | 0x100000)) << 32 | unsigned(__double2loint(g))) << 11;
  const int sh = 1023 + k - ev - f.x;  // at least 0 by the choice of k
  const unsigned long long p = __umul64hi(m, f.m);
  const long long r = ev == 0 || sh > 64 ? 0ll : sh <= 0 ? (long long)p : (long long)(((p >> (sh - 1)) + 1) >> 1);
  return fx_limbs((hi < 0 ? -r : r) + kFxHalf);
}

// One block per element: its exponent, then the limbs of alpha G with alpha = 2^(62-k) c, where c in
// [1, 2) and 2^ce are mantissa and exponent of the tables' scales (their chain): one unit of the element's
// result is then exactly 2^(k+ce) units of its input.  The factors come with their quadrature weights, which fw
// divides out: 64-bit integer products, since some 75 FP64 operations a point took 3.5 ms at N = 7,
// 32^3 elements (0.4 ms now, of which the bytes are 0.25), and ceedbp_set_kappa pays them on every call.
// NF = 6: stiffness factors G [e][6][q^3] -> [e][k][3][q^2] pairs of entries (00,01), (02,11), (12,22); NF = 1: mass factors.
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
__device__ __forceinline__ int fx_ratio_bits(int big, int small) {  // the ratio is below 2^this
  return (big >> 20) - (small >> 20) + ((big & 0xfffff) >= (small & 0xfffff));
}
__device__ __forceinline__ int fx_reach(int big, int small, int budget) {
  const int s = fx_ratio_bits(big, small);
  return s > kFxSpread ? 0 : max(budget + 1 - s, 0);
}

template <int NF>
__global__ void fx_factors_kernel(const double* __restrict__ G, const FxWeight* __restrict__ fw, int q, int ce, int colloc,
                                  int all_dirs, int budget, void* out, int* __restrict__ gexp) {
  constexpr int NR = NF == 6 ? 5 : 2;  // largest row sum; smallest of each direction and of the points' largest
  __shared__ int sred[NR][8];
  const int64_t e = blockIdx.x;
  const int q2 = q * q, q3 = q2 * q, tid = threadIdx.x;
  const double* Ge = G + e * NF * q3;
  int v[NR];
  v[0] = 0;
#pragma unroll
  for (int c = 1; c < NR; ++c) v[c] = 0x7fffffff;
  bool bad = false;
  for (int p = tid; p < q3; p += blockDim.x) {
    const FxWeight f = fw[p];
    int y[NF];
#pragma unroll
    for (int c = 0; c < NF; ++c) {
      const double g = Ge[size_t(c) * q3 + p];
      bad |= (__double2hiint(g) & 0x7ff00000) == 0x7ff00000;
      y[c] = fx_key(g, f);
    }
    if constexpr (NF == 6) {
      const int d = max(y[0], max(y[3], y[5])), top = max(d, max(y[1], max(y[2], y[4])));
      v[0] = max(v[0], max(fx_key_sum(y[0], y[1], y[2], top),
                           max(fx_key_sum(y[1], y[3], y[4], top), fx_key_sum(y[2], y[4], y[5], top))));
      v[1] = min(v[1], y[0]);
      v[2] = min(v[2], y[3]);
      v[3] = min(v[3], y[5]);
      v[4] = min(v[4], d);
    } else {
      v[0] = max(v[0], y[0] + 8);
      v[1] = min(v[1], y[0]);
    }
  }
  bad = __syncthreads_or(bad);
#pragma unroll
  for (int c = 0; c < NR; ++c) {
    v[c] = c == 0 ? __reduce_max_sync(0xffffffffu, v[c]) : __reduce_min_sync(0xffffffffu, v[c]);
    if ((tid & 31) == 0) sred[c][tid >> 5] = v[c];
  }
  __syncthreads();
  for (int i = 0; i < int(blockDim.x) / 32; ++i)
#pragma unroll
    for (int c = 0; c < NR; ++c) v[c] = c == 0 ? max(v[c], sred[c][i]) : min(v[c], sred[c][i]);
  int reach = 0;
  if (NF == 6 && colloc) {
    if (!all_dirs || fx_ratio_bits(v[0], min(v[1], min(v[2], v[3]))) <= 4)
#pragma unroll
      for (int d = 0; d < 3; ++d) reach |= fx_reach(v[0], v[1 + d], budget) << 4 * d;
  } else {
    reach = fx_reach(v[0], v[NR - 1], budget);
  }
  const int k = (v[0] >> 20) - 1021;  // the largest row sum is below 2^k: the rows of alpha G stay within 2^62
  // outside the grid: not finite, spread too far, or far from 1
  const bool off = bad || reach == 0 || k > 200 || k < -200;
  if (tid == 0) gexp[e] = off ? kFxNoGrid : (k + ce) * (1 << kFxReachBits) + reach;
  if (off) return;
  for (int p = tid; p < q3; p += blockDim.x) {
    const FxWeight f = fw[p];
    if constexpr (NF == 6) {
      int2 l[6];
#pragma unroll
      for (int c = 0; c < 6; ++c) l[c] = fx_factor(Ge[size_t(c) * q3 + p], f, k);
      int4* o = static_cast<int4*>(out) + e * 3 * q3 + size_t(p / q2) * 3 * q2 + p % q2;
#pragma unroll
      for (int c = 0; c < 3; ++c) o[size_t(c) * q2] = make_int4(l[2 * c].x, l[2 * c].y, l[2 * c + 1].x, l[2 * c + 1].y);
    } else {
      static_cast<int2*>(out)[e * q3 + p] = fx_factor(Ge[p], f, k);
    }
  }
}

}  // namespace

// Mantissa c of the chain over the weight of each point; returns the chain's exponent ce. 128-bit products of three
// 64-bit reciprocals: a long double operation per point took 3 ms at q = 17 where long double has 113 bits.
int fx_weights(const Basis1D& b, long double chain, std::vector<FxWeight>* out) {
  int ce = 0;
  const long double c = 2.0L * std::frexp(chain, &ce);  // chain = c 2^(ce-1)
  const int q = b.q;
  struct Recip {
    unsigned long long m;
    int x;  // m 2^(x-63)
  };
  std::vector<Recip> r(q), rc(q);
  auto recip = [](long double v) {
    int x = 0;
    const long double m = std::frexp(v, &x);  // in [1/2, 1)
    return Recip{(unsigned long long)std::ldexp(m, 64), x - 1};
  };
  for (int i = 0; i < q; ++i) {
    r[i] = recip(1.0L / b.w[i]);
    rc[i] = recip(c / b.w[i]);
  }
  typedef unsigned __int128 u128;
  out->resize(size_t(q) * q * q);
  FxWeight* f = out->data();
  for (int k = 0; k < q; ++k)
    for (int j = 0; j < q; ++j) {
      const u128 a = u128(rc[k].m) * r[j].m;
      const unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
      for (int i = 0; i < q; ++i, ++f) {
        u128 t = u128(hi) * r[i].m + ((u128(lo) * r[i].m) >> 64);  // all three over 2^64, at least 2^125
        int up = 0;
        for (; !(t >> 127); t <<= 1) ++up;
        *f = {(unsigned long long)(t >> 64), rc[k].x + r[j].x + r[i].x + 2 - up, 0};
      }
    }
  return ce - 1;
}

cudaError_t launch_fx_factors(const DeviceMesh& m, int kind, const double* G, void* out, int* gexp, cudaStream_t s) {
  const int q3 = m.q * m.q * m.q, threads = q3 >= 256 ? 256 : (q3 + 31) / 32 * 32;
  const int all_dirs = m.colloc && m.p1 <= 3, budget = m.p1 <= 4 ? 10 - m.p1 : 5;
  const FxWeight* fw = kind == kStiff ? m.fxw : m.fxmw;
  if (kind == kStiff)
    fx_factors_kernel<6><<<unsigned(m.nelem), threads, 0, s>>>(G, fw, m.q, m.fx->ce, m.colloc, all_dirs, budget, out, gexp);
  else
    fx_factors_kernel<1><<<unsigned(m.nelem), threads, 0, s>>>(G, fw, m.q, m.fx->mce, m.colloc, all_dirs, budget, out, gexp);
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
  if (b.colloc) {
    t->ce = fx_weights(b, t->chain, &t->weights);
    return;
  }
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
  t->ce = fx_weights(b, t->chain, &t->weights);
  t->mce = fx_weights(b, t->mchain, &t->mweights);
}

}  // namespace ceedbp
