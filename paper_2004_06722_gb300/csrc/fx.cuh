// Block fixed-point arithmetic of the FP64 element kernels.
//
// GB300 issues 2 FP64 FMAs per clock per SM but 64 widening integer
// multiply-adds (32 x 32 + 64 -> 64 bits; measured 64.4 per clock per SM), so an
// FP64 contraction is cheaper in integers: every value of an element is an
// integer on one power-of-two grid, 60 bits below the element's largest value,
// and a 1D product costs three widening multiply-adds per term instead of one
// FP64 FMA at 1/32 of their rate.
//
// Values.  x = h 2^31 + l with -2^30 <= l < 2^30 (two 32-bit limbs, "limbs" below) and |x| < 2^60.
// Matrix entries are M = h 2^31 + l likewise, scaled so that the largest absolute row sum is 2^62.
// A line product is
//   y = sum_j M_j x_j / 2^62 = HH + MM / 2^31,  HH = sum h_M h_x,  MM = sum (h_M l_x + l_M h_x)
// (the l l terms stay below one unit), so |y| < 2^60 again and the next stage starts without
// renormalisation.  MM / 2^31 is applied as twice MM's rounded upper word (one more multiply-add).
// The sums are integer sums: exact, and independent of their order; a sum of zeros is zero.
//
// Accuracy.  One unit is 2^-60 of an a-priori bound of a stage's values, against FP64's 2^-53 of each
// partial sum.  The bound of a derivative (the largest row sum of |D|) can exceed the actual values by
// 2^8; the gradient keeps enough bits for that, but the fluxes G grad u are moved up to 2^60 again by
// the element's actual maximum before the transposes, so that the two derivatives' slack does not add
// up (fx_limbs_up).  With that the error of one application on even elements, against quad-precision
// references, is 0.9-1.2 of that of the FP64 kernels this arithmetic replaces.  Values a grid cannot hold
// (infinities, NaN, elements whose factors spread over more than 2^5 (fx_setup.cu), exponents near the ends
// of the FP64 range) and uneven elements (below) take the FP64 form of the same kernel (the double overloads).
#pragma once

#include "common.cuh"
#include "df.cuh"

namespace ceedbp {

// Even-odd form of a centro-(anti)symmetric NO x NI matrix (Eq. (37)): e, o hold
// (M_ij + M_ij')/2 and (M_ij - M_ij')/2 for the first NO/2 rows (j' = NI-1-j; the middle column of
// an odd NI is held whole in e), m the middle row of an odd NO (over x+ or, antisymmetric, x-).
template <int NI, int NO, typename T>
struct EoMat {
  static constexpr int H = NI / 2, HC = (NI + 1) / 2, R = NO / 2;
  T e[R][HC];
  T o[R][H];
  T m[NO % 2 ? HC : 1];
};

constexpr long long kFxHalf = 1ll << 30;   // half a unit of h: limbs are taken from y + kFxHalf
constexpr long long kFxRound = 1ll << 31;  // MM starts here: its upper word is rounded to nearest, zeros stay zero

__device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }

// limbs of y, given y + kFxHalf
__device__ __forceinline__ int2 fx_limbs(long long yb) {
  return make_int2(int(yb >> 31), (int(yb) & 0x7fffffff) - int(kFxHalf));
}

// limbs of y 2^s, 0 <= s <= 30, |y 2^s| < 2^60, given y + (kFxHalf >> s)
__device__ __forceinline__ int2 fx_limbs_up(long long yb, int s) {
  return make_int2(int(__funnelshift_r(unsigned(yb), unsigned(yb >> 32), 31 - s)),
                   (int(unsigned(yb) << s) & 0x7fffffff) - int(kFxHalf));
}

// HH + MM / 2^31, MM started from kFxRound
__device__ __forceinline__ long long fx_join(long long hh, long long mm) { return fx_mad(int(mm >> 32), 2, hh); }

// limbs of v 2^(1082 - eb), below 2^60 in an element whose largest magnitude has the biased exponent eb
__device__ __forceinline__ int2 fx_from_double(double v, int eb) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int ev = (hi >> 20) & 0x7ff;
  const int d = min(eb - ev, 63);  // zeros and subnormals (ev = 0) shift out: eb is at least 500 here
  const unsigned long long mant =
      ((unsigned long long)(unsigned((hi & 0xfffff) | 0x100000)) << 32 | unsigned(lo)) << 7;
  const long long f = (long long)(mant >> d);
  return fx_limbs((hi < 0 ? -f : f) + kFxHalf);
}

// y = M x for one line, even-odd; emit(i, y_i), in limbs' arithmetic y_i + BIAS (int2 overload).
template <long long BIAS, int NI, int NO, bool ANTI, class Emit>
__device__ __forceinline__ void eo_line(const EoMat<NI, NO, int2>& M, const int2 (&x)[NI], Emit&& emit) {
  constexpr int H = NI / 2, HC = (NI + 1) / 2, R = NO / 2;
  int2 p[HC], q[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    p[j] = make_int2(x[j].x + x[NI - 1 - j].x, x[j].y + x[NI - 1 - j].y);
    q[j] = make_int2(x[j].x - x[NI - 1 - j].x, x[j].y - x[NI - 1 - j].y);
  }
  if constexpr (HC > H) p[H] = x[H];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    long long he = BIAS, me = kFxRound, ho = 0, mo = kFxRound;
#pragma unroll
    for (int j = 0; j < HC; ++j) {
      he = fx_mad(M.e[i][j].x, p[j].x, he);
      me = fx_mad(M.e[i][j].x, p[j].y, me);
      me = fx_mad(M.e[i][j].y, p[j].x, me);
    }
#pragma unroll
    for (int j = 0; j < H; ++j) {
      ho = fx_mad(M.o[i][j].x, q[j].x, ho);
      mo = fx_mad(M.o[i][j].x, q[j].y, mo);
      mo = fx_mad(M.o[i][j].y, q[j].x, mo);
    }
    const long long se = fx_join(he, me), so = fx_join(ho, mo);
    emit(i, se + so);
    emit(NO - 1 - i, ANTI ? so - se + 2 * BIAS : se - so);
  }
  if constexpr (NO % 2) {
    long long hh = BIAS, mm = kFxRound;
#pragma unroll
    for (int j = 0; j < (ANTI ? H : HC); ++j) {
      const int2 v = ANTI ? q[j < H ? j : 0] : p[j];
      hh = fx_mad(M.m[j].x, v.x, hh);
      mm = fx_mad(M.m[j].x, v.y, mm);
      mm = fx_mad(M.m[j].y, v.x, mm);
    }
    emit(R, fx_join(hh, mm));
  }
}

template <long long BIAS, int NI, int NO, bool ANTI, class Emit>
__device__ __forceinline__ void eo_line(const EoMat<NI, NO, double>& M, const double (&x)[NI], Emit&& emit) {
  constexpr int H = NI / 2, HC = (NI + 1) / 2, R = NO / 2;
  double p[HC], q[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    p[j] = x[j] + x[NI - 1 - j];
    q[j] = x[j] - x[NI - 1 - j];
  }
  if constexpr (HC > H) p[H] = x[H];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    // the odd half-sum on top of the even one: y_i comes out of the chain, its mirror is one more fma
    double se = __dmul_rn(M.e[i][0], p[0]);
#pragma unroll
    for (int j = 1; j < HC; ++j) se = __fma_rn(M.e[i][j], p[j], se);
    double s = se;
#pragma unroll
    for (int j = 0; j < H; ++j) s = __fma_rn(M.o[i][j], q[j], s);
    emit(i, s);
    emit(NO - 1 - i, ANTI ? __fma_rn(-2.0, se, s) : __fma_rn(2.0, se, -s));
  }
  if constexpr (NO % 2) {
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < (ANTI ? H : HC); ++j) s = __fma_rn(M.m[j], ANTI ? q[j < H ? j : 0] : p[j], s);
    emit(R, s);
  }
}

// One row of the geometric factors times the gradient at a point.
__device__ __forceinline__ long long fx_dot3(int2 a, int2 x, int2 b, int2 y, int2 c, int2 z) {
  long long hh = fx_mad(a.x, x.x, 0), mm = fx_mad(a.x, x.y, kFxRound);
  mm = fx_mad(a.y, x.x, mm);
  hh = fx_mad(b.x, y.x, hh);
  mm = fx_mad(b.x, y.y, mm);
  mm = fx_mad(b.y, y.x, mm);
  hh = fx_mad(c.x, z.x, hh);
  mm = fx_mad(c.x, z.y, mm);
  mm = fx_mad(c.y, z.x, mm);
  return fx_join(hh, mm);
}

// Largest magnitude of FP64 values by upper words; zero only if every value is zero (a subnormal whose upper
// word is zero counts as one).
struct FxTop {
  unsigned hi = 0, lo = 0;
  __device__ __forceinline__ void see(double v) {
    hi = max(hi, unsigned(__double2hiint(v)) & 0x7fffffffu);
    lo |= unsigned(__double2loint(v));
  }
  __device__ __forceinline__ unsigned top() const { return max(hi, min(lo, 1u)); }
};

// Uneven elements.  One unit of a stage is 2^-60 of the element's largest values, so a small entry of the
// result is as accurate as FP64's only while something of that size takes part in it: FP64's error is
// proportional to (|A| |u|)_i.  Every node is therefore asked for one of the three lines of nodes through it whose
// largest value reaches 2^-r of the element's (r from its factors, fx_setup.cu); an element with a node
// that has none (single peaks, values that fall by orders of magnitude) runs in FP64.  Nodes of the Dirichlet boundary
// whose results nobody reads are not asked.  With that every entry is within a few units of
// 2^-53 (|A| |u|)_i, as in FP64; without it the error was 2^-60 of the largest entry's scale.

// The word of a stage's largest magnitude that says so: the check needs no barrier of its own.  What it costs
// where elements are even: 0.8 % of a BP5 iteration at N = 7, 32^3 elements, nothing of BP3's (25^3), 1.3 % of BP1's
// at N = 3.  At N = 15 the elements along the edges of a Dirichlet boundary are uneven (values fall with the
// distance of the first node from two faces): 7 % of BP5, 10^3 elements.
constexpr unsigned kFxUneven = 0x80000000u;

// The smallest upper word that reaches (any value of an element of zeros).
__device__ __forceinline__ int fx_reach_word(unsigned top, int r, int slack = 0) {
  return r == 0 ? 0x7fffffff : max(int(top) - ((r + slack) << 20), 0);
}

// More bits that a line may lie below in a CG iteration: those by which the residual has fallen below the right-hand
// side.  An error of A p counts against b, not against p: CG reaches the same residual while the products'
// relative error stays below eps norm(b) / norm(r) (inexact Krylov methods: van den Eshof and Sleijpen, SIAM J. Matrix
// Anal. Appl. 26, 2004; Simoncini and Szyld, SIAM J. Sci. Comput. 25, 2003).  Late directions of BP1 span the
// quadrature weights: without these bits its solves went over to FP64 from order 9 on (N = 15: 8.0e9 instead of
// 1.8e10 DOFs/s).  True residuals reached from tolerance 1e-13, right-hand sides of random values, BP1 N = 15: 2.7e-14 as with
// FP64 kernels; with every direction on the grid 1.5e-13.
__device__ __forceinline__ int fx_slack(const SolveState* st, int c) {
  if (st == nullptr) return 0;
  const int d = (__double2hiint(st->c[c].bb) >> 20) - (__double2hiint(st->c[c].rr) >> 20);  // of squares, not negative
  return min(max(d >> 1, 0), 12);
}

// Whether one of the N values of a line reaches (the middle one first: most lines are answered by it).
template <int N>
__device__ __forceinline__ bool fx_line_reaches(const double* line, int step, int word) {
  auto at = [&](int n) { return __double2hiint(line[n * step]) & 0x7fffffff; };
  if (at(N / 2) >= word) return true;
  int t = 0;
#pragma unroll 4
  for (int n = 0; n < N; ++n) t = max(t, at(n));
  return t >= word;
}

// Where the threads of an element exchange the largest magnitude of a stage's values: one word for each
// stage, `step` words apart.
struct FxNorm {
  unsigned lanes;  // the warp's lanes of this element
  bool lead;       // one of them in each warp (false for threads without an element)
  unsigned* top;
  int step;
};

// The two arithmetics of the element kernels: L a stage's input, Raw its output.  see() collects the
// magnitudes (by upper words) of raw values that the next stage reads with load(); publish() before and
// take() after a barrier turn the element's largest into the shift that moves it up to 2^60.  take() is true
// if the word says that the block's elements are to run in FP64 (kFxUneven, larger than any magnitude).
struct FxArith {
  using L = int2;
  using Raw = long long;
  static constexpr long long kBias = kFxHalf;
  int hi = 0, lo = 0;
  int shift = 0, total = 0;
  long long bias = 0;  // kFxHalf on the unshifted grid
  __device__ __forceinline__ static L limbs(long long yb) { return fx_limbs(yb); }  // of a biased output
  __device__ __forceinline__ L load(Raw y) const { return fx_limbs_up(y + bias, shift); }
  __device__ __forceinline__ void see(Raw y) {
    const int w = int(y >> 32);
    hi = max(hi, w);
    lo = min(lo, w);
  }
  __device__ __forceinline__ void publish(const FxNorm& n, int stage) {
    const unsigned t = __reduce_max_sync(n.lanes, unsigned(max(hi, ~lo)));
    if (n.lead) atomicMax(n.top + stage * n.step, t);
    hi = lo = 0;
  }
  __device__ __forceinline__ bool take(const FxNorm& n, int stage) {
    const unsigned t = n.top[stage * n.step];
    shift = min(max(__clz(int(t)) - 4, 0), 30);
    total += shift;
    bias = kFxHalf >> shift;
    return t >= kFxUneven;
  }
};
struct F64Arith {
  using L = double;
  using Raw = double;
  static constexpr long long kBias = 0;
  int total = 0;
  __device__ __forceinline__ static L limbs(double y) { return y; }
  __device__ __forceinline__ L load(Raw y) const { return y; }
  __device__ __forceinline__ void see(Raw) {}
  __device__ __forceinline__ void publish(const FxNorm&, int) {}
  __device__ __forceinline__ bool take(const FxNorm&, int) { return false; }
};

// asynchronous copy of one double, or of zero
__device__ __forceinline__ void cp_async8_or_zero(void* dst, const void* src, bool zero) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(unsigned(__cvta_generic_to_shared(dst))), "l"(src),
               "r"(zero ? 0 : 8)
               : "memory");
}
__device__ __forceinline__ void l2_prefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Host: blocks of a kernel resident on the GPU (0: it does not fit), and the attribute that lets it use its
// shared memory.
inline int fx_resident(const void* kernel, int threads, size_t smem) {
  int dev = 0, sms = 0, nb = 0;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess ||
      cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, threads, smem) != cudaSuccess)
    return 0;
  return nb * sms;
}

// Host: SMs of the GPU, found once.
inline int fx_sms() {
  static const int n = [] {
    int dev = 0, sms = 0;
    return cudaGetDevice(&dev) == cudaSuccess &&
                   cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess
               ? sms
               : 0;
  }();
  return n;
}

// Host: elements in a slot's sequence such that one wave of resident blocks covers the mesh.
inline int fx_seq(int64_t nelem, int per_block, int resident) {
  const int64_t full = (nelem + per_block - 1) / per_block, res = resident < 1 ? 1 : resident;
  const int64_t n = (full + res - 1) / res;
  return int(n < kFxMaxSeq ? n : kFxMaxSeq);
}

}  // namespace ceedbp
