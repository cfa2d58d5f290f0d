// FP64 BK1..BK4 element kernel (Gauss quadrature, q = p1 + 1) in block fixed-point arithmetic
// (fx.cuh), in the interpolate-then-differentiate form of Eqs. (31)-(33) and Eq. (34).
//
// One thread per line, as in elem_fx.cuh, a q x q group of threads per element; all stages work in
// place in padded q^3 tiles (planes of q rows of q|1 values):
//
//   u (FP64, from the prefetch buffer) -> largest magnitude of the element -> limbs, tile A
//   x lines (j, k), y lines (q_x, k), z columns (q_x, q_y): J, tile A
//   stiffness: r lines A -> B, s lines A -> C, then the t column in A (Dq); G per point; Dq^T in
//     place in B, C, A; the three summed per column
//   mass: the mass factors per column
//   z, y, x lines: J^T, tile A, and the result in FP64
//
// The element's largest magnitude is moved up to 2^60 again (fx.cuh) after the interpolation, after the
// factors and after the sum: the row sums of J, Dq, Dq^T and J^T add up to 2^19 at N = 15, and without
// this the error would be up to 5 times the FP64 kernel's from N = 8 on.
//
// Quadrature weights: the factors are stored without the weights of their point, Dq^T and J^T are
// W^-1 Dq^T W and s^-1 J^T W (W: Gauss weights; s_i = sum_q |J_qi| w_q, which makes every row sum one),
// and the result of node (i, j, k) is multiplied by s_i s_j s_k in FP64 at the end, for the reason given
// in elem_fx.cuh.  The three directions of Dq^T have a quarter of the range each, so that their sum is
// in range.
//
// The FP32-pair arithmetic of BP1 and BP3 runs this kernel too, with pairs in and out: it is both closer to
// FP64 and faster than sums of pairs were (BK3, N = 5, 27 x 25 x 23 elements: 261 -> 200 us;
// BK1, N = 7, 32^3: 782 -> 485 us; one application's error 5 to 100 times smaller).
//
// Element sequences, prefetches and the FP64 form of elements off the grid: as in elem_fx.cuh.  The Helmholtz
// operator (Eq. (17)) is two launches, the second a mass operator that adds beta times its result: both in fixed
// point (one CG iteration, N = 7, 14^3 elements: 187 us, one FP64 pass that added the term at the quadrature points 458;
// N = 11, 9^3: 219 against 486; N = 7, 4^3: 40 against 44).
#pragma once

#include <algorithm>
#include <cstring>

#include "fx.cuh"

namespace ceedbp {

template <int P1>
struct FxGlTab {
  static constexpr int Q = P1 + 1;
  EoMat<P1, Q, int2> J;
  EoMat<Q, P1, int2> JT;
  EoMat<Q, Q, int2> D, DT;
  EoMat<P1, Q, double> J64;
  EoMat<Q, P1, double> JT64;
  EoMat<Q, Q, double> D64, DT64;
  double w[P1];  // s_i
};

template <int P1, int KIND>
struct FxGlShape {
  static constexpr int Q = P1 + 1, QQ = Q * Q, Q3 = QQ * Q, P3 = P1 * P1 * P1;
  static constexpr int S = Q | 1, PS = Q * S, TILE = Q * PS;  // 8-byte values
  static constexpr int NPT = (P3 + QQ - 1) / QQ;              // nodes of a thread
  static constexpr int EB = Q == 3 ? 14 : Q == 4 ? 8 : Q == 5 ? 5 : Q == 6 ? 7 : Q == 7 ? 5 : 1;  // as FxCoShape::EB
  static constexpr int NT = (EB * QQ + 31) / 32 * 32;
  static constexpr int NU = KIND == kStiff && Q >= 14 ? 1 : 2;  // u buffers, as FxCoShape::NU
  // the three directions share one loop body from q = 8 on (BK3, N = 6, 30^3 elements: 467 us rolled, 593 unrolled)
  static constexpr int UNROLL = Q >= 8 ? 1 : 3;
  static constexpr size_t SLOT = 8 * (size_t(NU) * P3 + (KIND == kStiff ? 3 : 1) * size_t(TILE));
  static constexpr size_t HEAD = 8 * 96 + 32 * size_t(EB);
  static constexpr size_t SMEM = HEAD + EB * SLOT;
  // Blocks per SM the registers are limited for, as FxCoShape::MINB. Spilled bytes a thread: BK3 40 at N = 7 (seven blocks,
  // 80 registers; six blocks 714 us against 597, 25^3 elements), 108 at 8, 350-440 at 10, 12 and 13, 250 at 15; BK1 up to 24
  // to N = 8, 140-160 at 10 to 13, 1150 at 14.
  static constexpr int BY_SMEM = int((size_t(227) << 10) / (SMEM + 1024)),
                       BY_REGS = 65536 / (NT * (KIND == kMass || Q <= 7 ? 80 : 96));
  static constexpr int MINB = BY_SMEM < BY_REGS ? BY_SMEM : BY_REGS < 1 ? 1 : BY_REGS;
};

// One element in arithmetic Ar, u in tile A.  factors: gradient to flux at point z of the own column, or
// value to value with the mass factors; done(shift) comes with the number of bits the values were moved up; out(i, y) turns the nodal results of line
// (j, k) = t into FP64, left in tile A.  weak(l) sees the values of line (j, k); if it
// is, uneven() may set the first stage's word to kFxUneven: false is then returned, with only the tiles overwritten.
template <int P1, int KIND, class Ar, class TJ, class TJT, class TD, class Weak, class Uneven, class Factors, class Mid,
          class Done, class Out>
__device__ __forceinline__ bool fx_gl_stages(void* tiles, int t, bool live, const TJ& J, const TJT& JT, const TD& D,
                                             const TD& DT, const FxNorm& norm, Weak&& weak, Uneven&& uneven, Factors&& factors,
                                             Mid&& mid, Done&& done, Out&& out) {
  using Sh = FxGlShape<P1, KIND>;
  using L = typename Ar::L;
  using Raw = typename Ar::Raw;
  constexpr int Q = Sh::Q, S = Sh::S, PS = Sh::PS, TILE = Sh::TILE;
  L* A = static_cast<L*>(tiles);
  Raw* Ax = static_cast<Raw*>(tiles);
  const int ti = t % Q, tj = t / Q;
  const int own = tj * S + ti;                  // column (q_x, q_y) = (ti, tj), step PS
  const int xb = (t / P1) * PS + (t % P1) * S;  // line (j, k) = (t % p1, t / p1), step 1
  const int yb = tj * PS + ti;                  // line (q_x, k) = (ti, tj), step S
  const bool xl = live && t < P1 * P1, yl = live && t < Q * P1;
  Ar ar;
  bool off = false;
  if (xl) {
    L l[P1];
#pragma unroll
    for (int n = 0; n < P1; ++n) l[n] = A[xb + n];
    off = weak(l);
    eo_line<Ar::kBias, P1, Q, false>(J, l, [&](int n, auto y) { A[xb + n] = Ar::limbs(y); });
  }
  __syncthreads();
  if (off) uneven();
  if (yl) {
    L l[P1];
#pragma unroll
    for (int n = 0; n < P1; ++n) l[n] = A[yb + n * S];
    eo_line<Ar::kBias, P1, Q, false>(J, l, [&](int n, auto y) { A[yb + n * S] = Ar::limbs(y); });
  }
  __syncthreads();
  if constexpr (KIND == kStiff) {
    if (live) {
      L l[P1];
#pragma unroll
      for (int n = 0; n < P1; ++n) l[n] = A[own + n * PS];
      eo_line<0, P1, Q, false>(J, l, [&](int n, auto y) {
        ar.see(y);
        Ax[own + n * PS] = y;
      });
    }
    Raw *Bx = Ax + TILE, *Cx = Bx + TILE;
    const L *B = A + TILE, *C = B + TILE;
    const int rb = tj * PS + ti * S;  // r: line (q_y, z) = (ti, tj), step 1;  s: line (q_x, z) = (ti, tj), step S
    ar.publish(norm, 1);
    __syncthreads();
    if (ar.take(norm, 1)) return false;
#pragma unroll Sh::UNROLL
    for (int dir = 0; dir < 3; ++dir) {
      if (dir == 2) __syncthreads();  // r and s have read tile A: t goes in place
      if (live) {
        const int base = dir == 0 ? rb : dir == 1 ? yb : own, step = dir == 0 ? 1 : dir == 1 ? S : PS;
        L* dst = A + (dir == 2 ? 0 : (dir + 1) * TILE) + base;
        L l[Q];
#pragma unroll
        for (int n = 0; n < Q; ++n) l[n] = ar.load(Ax[base + n * step]);
        eo_line<Ar::kBias, Q, Q, true>(D, l, [&](int n, auto y) { dst[n * step] = Ar::limbs(y); });
      }
    }
    mid();
    if (live) {
#pragma unroll 4
      for (int z = 0; z < Q; ++z) {
        Raw fr, fs, ft;
        factors(z, B[own + z * PS], C[own + z * PS], A[own + z * PS], fr, fs, ft);
        ar.see(fr);
        ar.see(fs);
        ar.see(ft);
        Bx[own + z * PS] = fr;
        Cx[own + z * PS] = fs;
        Ax[own + z * PS] = ft;
      }
    }
    ar.publish(norm, 2);
    __syncthreads();
    ar.take(norm, 2);
    if (live) {
#pragma unroll Sh::UNROLL
      for (int dir = 0; dir < 3; ++dir) {
        const int base = dir == 0 ? rb : dir == 1 ? yb : own, step = dir == 0 ? 1 : dir == 1 ? S : PS;
        Raw* dst = Ax + (dir == 2 ? 0 : (dir + 1) * TILE) + base;
        L l[Q];
#pragma unroll
        for (int n = 0; n < Q; ++n) l[n] = ar.load(dst[n * step]);
        eo_line<0, Q, Q, true>(DT, l, [&](int n, auto y) { dst[n * step] = y; });
      }
    }
    __syncthreads();
    if (live) {
#pragma unroll
      for (int z = 0; z < Q; ++z) {
        const Raw v = Bx[own + z * PS] + Cx[own + z * PS] + Ax[own + z * PS];
        ar.see(v);
        Ax[own + z * PS] = v;
      }
    }
  } else {
    mid();
    if (live) {
      L l[P1];
#pragma unroll
      for (int n = 0; n < P1; ++n) l[n] = A[own + n * PS];
      eo_line<Ar::kBias, P1, Q, false>(J, l, [&](int n, auto y) {
        const Raw v = factors(n, Ar::limbs(y));
        ar.see(v);
        Ax[own + n * PS] = v;
      });
    }
  }
  ar.publish(norm, 3);
  __syncthreads();
  if (ar.take(norm, 3) && KIND == kMass) return false;
  done(ar.total);
  if (live) {
    L l[Q];
#pragma unroll
    for (int z = 0; z < Q; ++z) l[z] = ar.load(Ax[own + z * PS]);
    eo_line<Ar::kBias, Q, P1, false>(JT, l, [&](int n, auto y) { A[own + n * PS] = Ar::limbs(y); });
  }
  __syncthreads();
  if (yl) {
    L l[Q];
#pragma unroll
    for (int n = 0; n < Q; ++n) l[n] = A[yb + n * S];
    eo_line<Ar::kBias, Q, P1, false>(JT, l, [&](int n, auto y) { A[yb + n * S] = Ar::limbs(y); });
  }
  __syncthreads();
  if (xl) {
    L l[Q];
#pragma unroll
    for (int n = 0; n < Q; ++n) l[n] = A[xb + n];
    double* W = static_cast<double*>(tiles) + xb;
    eo_line<0, Q, P1, false>(JT, l, [&](int n, auto y) { W[n] = out(n, y); });
  }
  __syncthreads();
  return true;
}

// PAIR: u and w^e are FP32 pairs (df.cuh; u may be FP64 as well), converted in shared memory.
// ADD: a.wl += a.beta w^e.
template <int P1, int NC, int KIND, bool PAIR, bool ADD>
__global__ void __launch_bounds__(FxGlShape<P1, KIND>::NT, FxGlShape<P1, KIND>::MINB)
    elem_fxgl_kernel(const DeviceMesh m, const ElemArgs a, const __grid_constant__ FxGlTab<P1> tab, const int ns) {
  using Sh = FxGlShape<P1, KIND>;
  constexpr int QQ = Sh::QQ, Q3 = Sh::Q3, P3 = Sh::P3, EB = Sh::EB, S = Sh::S, PS = Sh::PS, NPT = Sh::NPT;
  constexpr int NF = KIND == kStiff ? 6 : 1;
  extern __shared__ __align__(16) double smem_fx[];
  double* red = smem_fx;                                   // 32 * NC
  unsigned* smax = reinterpret_cast<unsigned*>(red + 96);  // [u, stage 1, 2, 3][2][EB]
  const int tid = threadIdx.x;
  const int slot = tid / QQ, t = tid - slot * QQ;
  const bool live = slot < EB;  // threads that pad the block to whole warps only take part in barriers
  double* ubuf = reinterpret_cast<double*>(reinterpret_cast<char*>(smem_fx) + Sh::HEAD + size_t(live ? slot : 0) * Sh::SLOT);
  double* tiles = ubuf + Sh::NU * P3;
  const void* fx = KIND == kStiff ? static_cast<const void*>(m.Gfx) : static_cast<const void*>(m.Mfx);
  const int* fxe = KIND == kStiff ? m.gexp : m.mexp;

  const int64_t e0 = int64_t(blockIdx.x) * (EB * ns);
  const int nblk = m.nelem - e0 < EB * ns ? int(m.nelem - e0) : EB * ns;
  const int nit = (nblk + EB - 1) / EB * NC;
  // the slot's element of item `it` (a slot past the block's last element repeats that one, unstored)
  auto elem_of = [&](int it) { return e0 + min((it / NC) * EB + slot, nblk - 1); };
  const unsigned lanes = __match_any_sync(0xffffffffu, slot);  // the warp's lanes of this slot
  const bool lead = live && (tid & 31) == __ffs(int(lanes)) - 1;
  auto place = [](int idx) { return idx / (P1 * P1) * PS + idx / P1 % P1 * S + idx % P1; };  // of a node in a tile

  // whether the thread has an n-th node (known to the compiler for all but the last)
  auto has = [&](int n) { return (n + 1) * QQ <= P3 || t + n * QQ < P3; };
  int g[NPT];
  unsigned dnext = 0, dcur = 0;  // Dirichlet bits of the thread's nodes
  auto load_l2g = [&](int it) {
    const int* l2g = m.l2g + elem_of(it) * P3;
#pragma unroll
    for (int n = 0; n < NPT; ++n)
      if (has(n)) g[n] = __ldg(l2g + t + n * QQ);
  };
  auto fetch_u = [&](int it) {
    double* dst = ubuf + (it % Sh::NU) * P3;
    const double* src = (PAIR && a.u == nullptr ? reinterpret_cast<const double*>(a.u_df) : a.u) + (NC == 1 ? 0 : it % NC);
    dnext = 0;
#pragma unroll
    for (int n = 0; n < NPT; ++n) {
      if (!has(n)) continue;
      const int gg = g[n] ^ (g[n] >> 31);  // -(g + 1) for Dirichlet nodes
      dnext |= unsigned(g[n] < 0) << n;
      cp_async8_or_zero(dst + t + n * QQ, src + size_t(gg) * NC, g[n] < 0 && a.mask_in);
    }
  };
  auto prefetch_factors = [&](int64_t e) {
    const char* G = (fx != nullptr ? static_cast<const char*>(fx) : reinterpret_cast<const char*>(a.G)) + e * (8 * NF * Q3);
    for (int b = t * 128; b < 8 * NF * Q3; b += QQ * 128) l2_prefetch(G + b);
  };
  for (int i = tid; i < 8 * EB; i += Sh::NT) smax[i] = 0u;
  if (live) {
    load_l2g(0);
    prefetch_factors(elem_of(0));
  }
  if (a.state != nullptr && a.state->stop) return;  // read beside the map
  if (live) fetch_u(0);
  double dot[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) dot[c] = 0.0;
  const double wjk = live && t < P1 * P1 ? tab.w[t % P1] * tab.w[t / P1] : 0.0;
  __syncthreads();

#pragma unroll 1
  for (int it = 0; it < nit; ++it) {
    const int64_t e = elem_of(it);
    const bool store = live && (it / NC) * EB + slot < nblk;
    const int c = NC == 1 ? 0 : it % NC;
    double* su = ubuf + (it % Sh::NU) * P3;
    cp_async_wait_all();
    dcur = dnext;
    if (PAIR && a.u == nullptr && live) {
#pragma unroll
      for (int n = 0; n < NPT; ++n)
        if (has(n)) su[t + n * QQ] = df_to_f64(reinterpret_cast<const dfloat*>(su)[t + n * QQ]);
    }
    FxTop seen;
    if (live) {
#pragma unroll
      for (int n = 0; n < NPT; ++n)
        if (has(n)) seen.see(su[t + n * QQ]);
      if (it + 1 < nit) load_l2g(it + 1);
    }
    const unsigned mx = __reduce_max_sync(lanes, seen.top());
    const int code = live && fxe != nullptr ? __ldg(fxe + e) : kFxNoGrid, ge = code >> kFxReachBits;
    const FxNorm norm{lanes, lead, smax + (it & 1) * EB + (live ? slot : 0), 2 * EB};
    if (lead) atomicMax(norm.top, mx);
    __syncthreads();
    const unsigned top = live ? *norm.top : 0u;
    const int eb = top == 0u ? 1023 : int(top >> 20);  // every value is zero: any exponent
    const bool bad = live && (code == kFxNoGrid || eb < 500 || eb > 1500);
    if (t < 4 && live) smax[(2 * t + (~it & 1)) * EB + slot] = 0u;
    bool ahead = live && it + 1 < nit;
    auto mid = [&]() {  // once, also if the element changes to FP64
      if (ahead) {
        ahead = false;
        if (Sh::NU == 2) fetch_u(it + 1);
        if (NC == 1 || (it + 1) % NC == 0) prefetch_factors(elem_of(it + 1));
      }
    };
    if (live) {
#pragma unroll
      for (int n = 0; n < NPT; ++n)
        if (has(n)) reinterpret_cast<int2*>(tiles)[place(t + n * QQ)] = fx_from_double(su[t + n * QQ], eb);
    }
    bool f64 = __syncthreads_or(bad);
    if (!f64) {
      double sc = 0.0;
      // a line (j, k) below the limb of the smallest value that reaches, and its nodes one by one. Pairs carry 47
      // bits: they keep theirs at ratios up to 2^10 larger.
      const int reach = PAIR ? min((code & 15) + 10, 15) : code & 15;
      auto weak = [&](const int2(&l)[P1]) {
        int hi = 0, lo = 0;
#pragma unroll
        for (int n = 0; n < P1; ++n) {
          hi = max(hi, l[n].x);
          lo = min(lo, l[n].x);
        }
        return max(hi, ~lo) < int(((top & 0xfffffu) | 0x100000u) << 8 >> reach);
      };
      auto uneven = [&]() {
        const int* l2g = m.l2g + e * P3 + t * P1;
        bool free = !a.skip_dirichlet_out;  // lines of the Dirichlet boundary are the usual weak ones
#pragma unroll
        for (int i = 0; i < P1; ++i) free |= __ldg(l2g + i) >= 0;
        if (!free) return;
        const int slack = fx_slack(a.state, c), word = fx_reach_word(top, reach, slack), j = t % P1, k = t / P1;
        if (slack > 0 && fx_line_reaches<P1>(su + t * P1, 1, word)) return;
        bool off = false;
#pragma unroll 1
        for (int i = 0; i < P1; ++i)
          off |= !fx_line_reaches<P1>(su + k * P1 * P1 + i, P1, word) &&
                 !fx_line_reaches<P1>(su + j * P1 + i, P1 * P1, word) &&
                 !(a.skip_dirichlet_out && __ldg(l2g + i) < 0);
        if (off)
          for (int s = 0; s < EB; ++s) atomicMax(smax + ((KIND == kStiff ? 2 : 6) + (it & 1)) * EB + s, kFxUneven);
      };
      auto done = [&](int shift) { sc = wjk * __hiloint2double((eb + ge - shift - (1082 - 1023)) << 20, 0); };
      auto out = [&](int i, long long y) { return __ll2double_rn(y) * (tab.w[i] * sc); };
      if constexpr (KIND == kStiff) {
        const int4* G = m.Gfx + e * 3 * Q3 + t;
        f64 = !fx_gl_stages<P1, KIND, FxArith>(
            tiles, t, live, tab.J, tab.JT, tab.D, tab.DT, norm, weak, uneven,
            [&](int z, int2 r, int2 s, int2 tt, long long& fr, long long& fs, long long& ft) {
              const int4 g0 = __ldcs(G + (3 * z + 0) * QQ), g1 = __ldcs(G + (3 * z + 1) * QQ),
                         g2 = __ldcs(G + (3 * z + 2) * QQ);
              const int2 g00 = make_int2(g0.x, g0.y), g01 = make_int2(g0.z, g0.w), g02 = make_int2(g1.x, g1.y),
                         g11 = make_int2(g1.z, g1.w), g12 = make_int2(g2.x, g2.y), g22 = make_int2(g2.z, g2.w);
              fr = fx_dot3(g00, r, g01, s, g02, tt);
              fs = fx_dot3(g01, r, g11, s, g12, tt);
              ft = fx_dot3(g02, r, g12, s, g22, tt);
            },
            mid, done, out);
      } else {
        const int2* M = m.Mfx + e * Q3 + t;
        f64 = !fx_gl_stages<P1, KIND, FxArith>(
            tiles, t, live, tab.J, tab.JT, tab.D, tab.DT, norm, weak, uneven,
            [&](int z, int2 v) {
              const int2 f = __ldcs(M + z * QQ);
              long long mm = fx_mad(f.x, v.y, kFxRound);
              mm = fx_mad(f.y, v.x, mm);
              return fx_join(fx_mad(f.x, v.x, 0), mm);
            },
            mid, done, out);
      }
    }
    if (f64) {
      if (live) {
#pragma unroll
        for (int n = 0; n < NPT; ++n)
          if (has(n)) tiles[place(t + n * QQ)] = su[t + n * QQ];
      }
      __syncthreads();
      auto done = [](int) {};
      auto out = [](int, double y) { return y; };
      auto weak = [](const double(&)[P1]) { return false; };
      auto uneven = []() {};
      const double* G = a.G + e * NF * Q3 + t;
      if constexpr (KIND == kStiff) {
        fx_gl_stages<P1, KIND, F64Arith>(
            tiles, t, live, tab.J64, tab.JT64, tab.D64, tab.DT64, norm, weak, uneven,
            [&](int z, double r, double s, double tt, double& fr, double& fs, double& ft) {
              const double* Gz = G + z * QQ;
              const double g00 = __ldcs(Gz), g01 = __ldcs(Gz + Q3), g02 = __ldcs(Gz + 2 * Q3), g11 = __ldcs(Gz + 3 * Q3),
                           g12 = __ldcs(Gz + 4 * Q3), g22 = __ldcs(Gz + 5 * Q3);
              fr = g00 * r + g01 * s + g02 * tt;
              fs = g01 * r + g11 * s + g12 * tt;
              ft = g02 * r + g12 * s + g22 * tt;
            },
            mid, done, out);
      } else {
        fx_gl_stages<P1, KIND, F64Arith>(
            tiles, t, live, tab.J64, tab.JT64, tab.D64, tab.DT64, norm, weak, uneven,
            [&](int z, double v) { return __ldcs(G + z * QQ) * v; }, mid, done, out);
      }
    }
    // w^e to the local output (coalesced), (u^e, w^e)
    if (store) {
      double* wl = a.wl + size_t(e) * P3 * NC + c;
      double acc = 0.0;
#pragma unroll
      for (int n = 0; n < NPT; ++n) {
        if (!has(n)) continue;
        const int idx = t + n * QQ;
        double w = tiles[place(idx)];
        if (!(a.skip_dirichlet_out && ((dcur >> n) & 1u))) {
          if constexpr (ADD) w = wl[size_t(idx) * NC] + a.beta * w;
          if constexpr (PAIR) reinterpret_cast<dfloat*>(wl)[size_t(idx) * NC] = f64_to_df(w);
          else wl[size_t(idx) * NC] = w;
        }
        acc += w * su[idx];
      }
#pragma unroll
      for (int q = 0; q < NC; ++q)
        if (q == c) dot[q] += acc;
    }
    if (Sh::NU == 1 && live && it + 1 < nit) fetch_u(it + 1);  // the thread's values were read last above
  }
  if (a.partials != nullptr) cg_alpha<NC>(dot, a.partials, a.state, red);
}

template <int P1>
FxGlTab<P1> elem_fxgl_tab(const DeviceMesh& m) {
  FxGlTab<P1> t;
  const FxTables& f = *m.fx;
  std::memcpy(&t.J, f.J.data(), sizeof(t.J));
  std::memcpy(&t.JT, f.JT.data(), sizeof(t.JT));
  std::memcpy(&t.D, f.D.data(), sizeof(t.D));
  std::memcpy(&t.DT, f.DT.data(), sizeof(t.DT));
  std::memcpy(&t.J64, f.J64.data(), sizeof(t.J64));
  std::memcpy(&t.JT64, f.JT64.data(), sizeof(t.JT64));
  std::memcpy(&t.D64, f.D64.data(), sizeof(t.D64));
  std::memcpy(&t.DT64, f.DT64.data(), sizeof(t.DT64));
  std::memcpy(t.w, f.w.data(), sizeof(t.w));
  return t;
}

// Blocks resident on the GPU (0: the kernel does not fit), found once per instantiation; the
// attribute that lets it use its shared memory is set on the way.
template <int P1, int NC, int KIND, bool PAIR, bool ADD>
int elem_fxgl_resident() {
  using Sh = FxGlShape<P1, KIND>;
  static const int n = fx_resident(reinterpret_cast<const void*>(elem_fxgl_kernel<P1, NC, KIND, PAIR, ADD>), Sh::NT, Sh::SMEM);
  return n;
}

// Elements in a slot's sequence: one wave of resident blocks covers the mesh.
template <int P1, int NC, int KIND>
int elem_fxgl_seq(int64_t nelem) {
  return fx_seq(nelem, FxGlShape<P1, KIND>::EB, elem_fxgl_resident<P1, NC, KIND, false, false>());
}

template <int P1, int NC, int KIND>
int elem_fxgl_blocks_t(int64_t nelem) {
  const int64_t per = int64_t(FxGlShape<P1, KIND>::EB) * elem_fxgl_seq<P1, NC, KIND>(nelem);
  return int((nelem + per - 1) / per);
}

template <int P1, int NC, int KIND, bool PAIR = false, bool ADD = false>
cudaError_t launch_elem_fxgl_k(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s) {
  using Sh = FxGlShape<P1, KIND>;
  if (elem_fxgl_resident<P1, NC, KIND, PAIR, ADD>() < 1) return cudaErrorInvalidConfiguration;
  const int ns = elem_fxgl_seq<P1, NC, KIND>(m.nelem), blocks = elem_fxgl_blocks_t<P1, NC, KIND>(m.nelem);
  elem_fxgl_kernel<P1, NC, KIND, PAIR, ADD><<<blocks, Sh::NT, Sh::SMEM, s>>>(m, a, elem_fxgl_tab<P1>(m), ns);
  return cudaGetLastError();
}

template <int P1, int NC>
cudaError_t launch_elem_fxgl_n(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s) {
  if (kind == kMass) return launch_elem_fxgl_k<P1, NC, kMass>(m, a, s);
  if (a.beta == 0.0) return launch_elem_fxgl_k<P1, NC, kStiff>(m, a, s);
  ElemArgs stiff = a, mass = a;  // A u first; the mass pass adds beta B u and sums (u, w) of both
  stiff.partials = nullptr;
  mass.G = a.Mq;
  const cudaError_t e = launch_elem_fxgl_k<P1, NC, kStiff>(m, stiff, s);
  return e != cudaSuccess ? e : launch_elem_fxgl_k<P1, NC, kMass, false, true>(m, mass, s);
}

template <int P1>
cudaError_t launch_elem_fxgl_t(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s) {
  return m.ncomp == 3 ? launch_elem_fxgl_n<P1, 3>(m, kind, a, s) : launch_elem_fxgl_n<P1, 1>(m, kind, a, s);
}

template <int P1>
cudaError_t launch_elem_fxgl_pair_t(const DeviceMesh& m, int kind, const ElemArgs& a, cudaStream_t s) {
  return kind == kMass ? launch_elem_fxgl_k<P1, 1, kMass, true>(m, a, s)
                       : launch_elem_fxgl_k<P1, 1, kStiff, true>(m, a, s);
}

// Largest grid of the order's launches with m's elements (room for their partial sums).
template <int P1>
int elem_fxgl_blocks_any(const DeviceMesh& m) {
  if (m.ncomp == 3) return std::max(elem_fxgl_blocks_t<P1, 3, kStiff>(m.nelem), elem_fxgl_blocks_t<P1, 3, kMass>(m.nelem));
  return std::max(elem_fxgl_blocks_t<P1, 1, kStiff>(m.nelem), elem_fxgl_blocks_t<P1, 1, kMass>(m.nelem));
}

}  // namespace ceedbp
