// FP64 BK5/BK6 element kernel (collocated stiffness, Eq. (22) with J = I) in block fixed-point
// arithmetic (fx.cuh).
//
// One thread per line: a group of p1^2 threads (a slot) holds one element; thread (i, j) owns the
// column k = 0..p1-1 of every tile and, in the r and s stages, one line of the other two directions,
// so each 1D product is a whole line in one thread's registers, in even-odd form, with the matrix
// entries in the constant bank (every thread of a warp uses the same entry at the same time).
//
//   u column (FP64, from the prefetch buffer) -> largest magnitude of the element -> limbs, tile A
//   r lines A -> B, s lines A -> C, then the t column in place in A
//   G: (u_r, u_s, u_t) -> (w_r, w_s, w_t) per point, in place in B, C, A; their largest magnitude
//   in the element sets the shift they are read back with
//   r^T in place in B, s^T in C, t^T in A; the three summed per column
//
// Quadrature weights.  The factors are stored without the weights w_i w_j w_k of their point and the
// transposes use D_ni w_n / w_i, so that G grad u and what follows have the smooth spread of the
// metric (the weights alone span 2^10 at N = 7 and would cost the element's grid those bits at the
// corners); the result of node (i, j, k) is multiplied by w_i w_j w_k in FP64 at the end.
//
// Each slot works through a sequence of elements; l2g of the next element is loaded at the top of the
// current one, its u values are copied to shared memory (cp.async) once the gradient is done, and its
// factors are prefetched into L2, so that the dependent gather overlaps a whole element's arithmetic.
//
// An element whose values or factors do not fit the fixed-point grid or are too uneven for it (fx.cuh), and
// every element when the context holds no fixed-point factors, runs the same stages in FP64 (a.G, with weights).
// That form is not shaped for the FP64 pipe: 0.8 to 1.3 times the FP64 kernels that this one replaced, all
// elements in it (solves on 1.5e6 DOFs; N = 7 222 -> 246 us an iteration, N = 11 266 -> 340, N = 12 482 -> 390). Blocks of 256 threads
// of whole elements for it alone gained less than 10 % of that and lost elsewhere.
#pragma once

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "fx.cuh"

namespace ceedbp {

template <int P1>
struct FxCoTab {
  EoMat<P1, P1, int2> D, DT;
  EoMat<P1, P1, double> D64, DT64;
  double w[P1];   // GLL weights
};

// W: threads per column of an element: 1, or 3 on small meshes (elem_fx_wide). Three groups of p1^2 threads
// then take one direction's lines and every third point of the columns each: the same operations in the
// same order on every value, a shorter chain for one element, more barriers and less reuse for many.
template <int P1, int W = 1>
struct FxCoShape {
  static constexpr int PP = P1 * P1, P3 = PP * P1;
  static constexpr int S = P1 | 1;      // odd row length: lines of every direction are free of bank conflicts
  static constexpr int TILE = PP * S;   // 8-byte values
  // Elements per block.  One where p1^2 threads fill their warps: the element index is then the same for
  // the whole block and lives in uniform registers, and a barrier joins p1^2 threads only (N = 7,
  // E = 2^16: 704 -> 658 us against two elements per block; N = 8, E = 15625: 523 -> 337 us against
  // three).  Several where it would leave lanes idle (p1 = 6: 365 us with seven, 445 us with one, E = 40^3).
  static constexpr int EB = W == 3 ? 1 : P1 == 2 ? 32 : P1 == 3 ? 14 : P1 == 4 ? 8 : P1 == 5 ? 5 : P1 == 6 ? 7 : 1;
  static constexpr int NT = (EB * W * PP + 31) / 32 * 32;
  static constexpr int KC = (P1 + W - 1) / W;  // points of a column per thread
  // u buffers: the next element's values land while the current one is computed; from p1 = 13 to 15 one
  // buffer, filled between elements, lets one more block fit on the SM instead
  static constexpr int NU = P1 >= 13 && P1 <= 15 ? 1 : 2;
  // the three directions of a stage share one loop body from p1 = 14 on: unrolled, the code outgrows the
  // instruction cache (N = 14, E = 14^3: 524 us unrolled, 424 us rolled; N = 7: 350 against 366 us)
  static constexpr int UNROLL = P1 >= 14 ? 1 : 3;
  static constexpr size_t SLOT = 8 * (size_t(NU) * P3 + 3 * size_t(TILE));
  static constexpr size_t HEAD = 8 * 96 + 16 * size_t(EB);
  static constexpr size_t SMEM = HEAD + EB * SLOT;
  // Blocks per SM the registers are limited for: what shared memory holds, at 96 registers or more
  // (p1 = 8: eight blocks, 120 registers: 350 us at E = 2^15; ten, 96 registers: 370 us), that is five warps
  // on each of an SM's four partitions (N = 8, 20^3 elements, one iteration: seven blocks of three warps, 80 registers 284 us,
  // six 272 us). From N = 11 on the lines of a thread do not fit these registers: spilled bytes a thread 264 at N = 11,
  // 1172 at 12 (three blocks, 96 registers), 770-830 at 13 and 14, none at 15 (one block).
  static constexpr int BY_SMEM = int((size_t(227) << 10) / (SMEM + 1024)), BY_REGS = 4 * (512 / 96) / (NT / 32);
  static constexpr int MINB = W == 3 ? 1 : P1 == 8 ? 8 : BY_SMEM < BY_REGS ? BY_SMEM : BY_REGS;
};

// Per-thread view of one element of a slot.
template <int P1>
struct FxCoElem {
  int t, ti, tj, grp;  // grp: the direction group, 0 with one thread per column
  void* A;           // tiles A, B, C
  const double* su;  // the element's u, [k][t]
};

// Contractions and factors of one element in arithmetic Ar (FxArith or F64Arith), u in tile A.
// factors(k, gradient, flux) multiplies by G at point k of the own column; done(shift) comes with the
// number of bits the fluxes were moved up; out(k, r, s, t) receives the three transposes.
// False is returned, with only the tiles overwritten, if the element turned out uneven.
template <int P1, int W, class Ar, class Tab, class Factors, class Mid, class Done, class Out>
__device__ __forceinline__ bool fx_co_stages(const FxCoElem<P1>& el, const Tab& D, const Tab& DT, bool live,
                                             const FxNorm& norm, Factors&& factors, Mid&& mid, Done&& done, Out&& out) {
  using Sh = FxCoShape<P1, W>;
  using L = typename Ar::L;
  using Raw = typename Ar::Raw;
  constexpr int S = Sh::S, PS = P1 * S;
  L *A = static_cast<L*>(el.A), *B = A + Sh::TILE, *C = B + Sh::TILE;
  Raw *Ar_ = static_cast<Raw*>(el.A), *Br = Ar_ + Sh::TILE, *Cr = Br + Sh::TILE;
  // lines of thread t: r (j, k), base t S, step 1;  s (i, k), base k P1 S + i, step S;  t (i, j), the own column
  const int rb = el.t * S, sb = el.tj * PS + el.ti, own = el.tj * S + el.ti;
  Ar ar;
  if constexpr (W == 3) {
    const int dir = el.grp;
    const int base = dir == 0 ? rb : dir == 1 ? sb : own, step = dir == 0 ? 1 : dir == 1 ? S : PS;
    L l[P1];
    if (live) {
#pragma unroll
      for (int n = 0; n < P1; ++n) l[n] = A[base + n * step];
    }
    __syncthreads();  // t goes in place
    if (live) {
      L* dst = A + (dir == 2 ? 0 : (dir + 1) * Sh::TILE) + base;
      eo_line<Ar::kBias, P1, P1, true>(D, l, [&](int n, auto y) { dst[n * step] = Ar::limbs(y); });
    }
    __syncthreads();
  } else {
#pragma unroll Sh::UNROLL
    for (int dir = 0; dir < 3; ++dir) {
      if (dir == 2) __syncthreads();  // r and s have read tile A: t goes in place
      if (live) {
        const int base = dir == 0 ? rb : dir == 1 ? sb : own, step = dir == 0 ? 1 : dir == 1 ? S : PS;
        L* dst = A + (dir == 2 ? 0 : (dir + 1) * Sh::TILE) + base;
        L l[P1];
#pragma unroll
        for (int n = 0; n < P1; ++n) l[n] = A[base + n * step];
        eo_line<Ar::kBias, P1, P1, true>(D, l, [&](int n, auto y) { dst[n * step] = Ar::limbs(y); });
      }
    }
  }
  mid();
  if (live) {
#pragma unroll 4
    for (int k = el.grp; k < P1; k += W) {
      Raw fr, fs, ft;
      factors(k, B[own + k * PS], C[own + k * PS], A[own + k * PS], fr, fs, ft);
      ar.see(fr);
      ar.see(fs);
      ar.see(ft);
      Br[own + k * PS] = fr;
      Cr[own + k * PS] = fs;
      Ar_[own + k * PS] = ft;
    }
  }
  ar.publish(norm, 1);
  __syncthreads();
  if (ar.take(norm, 1)) return false;
  done(ar.total);
  if (live) {
#pragma unroll W == 3 ? 1 : Sh::UNROLL
    for (int dir = el.grp; dir < 3; dir += W == 3 ? 3 : 1) {
      const int base = dir == 0 ? rb : dir == 1 ? sb : own, step = dir == 0 ? 1 : dir == 1 ? S : PS;
      Raw* dst = Ar_ + (dir == 2 ? 0 : (dir + 1) * Sh::TILE) + base;
      L l[P1];
#pragma unroll
      for (int n = 0; n < P1; ++n) l[n] = ar.load(dst[n * step]);
      eo_line<0, P1, P1, true>(DT, l, [&](int n, auto y) { dst[n * step] = y; });
    }
  }
  __syncthreads();
  if (live) {
#pragma unroll
    for (int h = 0; h < Sh::KC; ++h) {
      const int k = W * h + el.grp;
      if (W == 1 || k < P1) out(h, k, Br[own + k * PS], Cr[own + k * PS], Ar_[own + k * PS]);
    }
  }
  return true;
}

template <int P1, int NC, bool HELM, int W>
__global__ void __launch_bounds__(FxCoShape<P1, W>::NT, FxCoShape<P1, W>::MINB)
    elem_fx_kernel(const DeviceMesh m, const ElemArgs a, const __grid_constant__ FxCoTab<P1> tab, const int ns) {
  using Sh = FxCoShape<P1, W>;
  constexpr int PP = Sh::PP, P3 = Sh::P3, EB = Sh::EB, S = Sh::S, PS = P1 * S, KC = Sh::KC;
  extern __shared__ __align__(16) double smem_fx[];
  double* red = smem_fx;                                  // 32 * NC
  unsigned* smax = reinterpret_cast<unsigned*>(red + 96);  // [u, fluxes][2][EB]
  const int tid = threadIdx.x;
  const int slot = tid / (W * PP);
  const bool live = slot < EB;  // threads that pad the block to whole warps only take part in barriers
  char* base = reinterpret_cast<char*>(smem_fx) + Sh::HEAD + size_t(live ? slot : 0) * Sh::SLOT;
  double* ubuf = reinterpret_cast<double*>(base);
  FxCoElem<P1> el;
  el.grp = W == 1 ? 0 : tid / PP % W;
  el.t = tid - (W * slot + el.grp) * PP;
  el.ti = el.t % P1;
  el.tj = el.t / P1;
  el.A = ubuf + Sh::NU * P3;

  const int64_t e0 = int64_t(blockIdx.x) * (EB * ns);
  const int nblk = m.nelem - e0 < EB * ns ? int(m.nelem - e0) : EB * ns;
  const int nit = (nblk + EB - 1) / EB * NC;
  // the slot's element of item `it` (a slot past the block's last element repeats that one, unstored)
  auto elem_of = [&](int it) { return e0 + min((it / NC) * EB + slot, nblk - 1); };
  const unsigned lanes = __match_any_sync(0xffffffffu, slot);  // the warp's lanes of this slot
  const bool lead = live && (tid & 31) == __ffs(int(lanes)) - 1;

  int g[KC];
  unsigned dnext = 0, dcur = 0;  // Dirichlet bits of the own column
  auto load_l2g = [&](int it) {
    const int* l2g = m.l2g + elem_of(it) * P3 + el.t;
#pragma unroll
    for (int h = 0; h < KC; ++h) g[h] = W == 1 || W * h + el.grp < P1 ? __ldg(l2g + (W * h + el.grp) * PP) : 0;
  };
  auto fetch_u = [&](int it) {
    double* dst = ubuf + (it % Sh::NU) * P3 + el.t;
    const double* src = a.u + (NC == 1 ? 0 : it % NC);
    dnext = 0;
#pragma unroll
    for (int h = 0; h < KC; ++h) {
      if (W > 1 && W * h + el.grp >= P1) continue;
      const int gg = g[h] ^ (g[h] >> 31);  // -(g + 1) for Dirichlet nodes
      dnext |= unsigned(g[h] < 0) << h;
      cp_async8_or_zero(dst + (W * h + el.grp) * PP, src + size_t(gg) * NC, g[h] < 0 && a.mask_in);
    }
  };
  auto prefetch_G = [&](int64_t e) {
    const char* G = m.Gfx != nullptr ? reinterpret_cast<const char*>(m.Gfx + e * 3 * P3)
                                     : reinterpret_cast<const char*>(a.G + e * 6 * P3);
    for (int b = (el.grp * PP + el.t) * 128; b < 48 * P3; b += W * PP * 128) l2_prefetch(G + b);
  };
  for (int i = tid; i < 4 * EB; i += Sh::NT) smax[i] = 0u;
  if (live) {
    load_l2g(0);
    prefetch_G(elem_of(0));
  }
  if (a.state != nullptr && a.state->stop) return;  // read beside the map
  if (live) fetch_u(0);
  double dot[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) dot[c] = 0.0;
  const double wij = live ? tab.w[el.ti] * tab.w[el.tj] : 0.0;
  __syncthreads();

#pragma unroll 1
  for (int it = 0; it < nit; ++it) {
    const int64_t e = elem_of(it);
    const bool store = live && (it / NC) * EB + slot < nblk;
    const int c = NC == 1 ? 0 : it % NC;
    el.su = ubuf + (it % Sh::NU) * P3 + el.t;
    cp_async_wait_all();
    dcur = dnext;
    FxTop seen;
    if (live) {
#pragma unroll
      for (int h = 0; h < KC; ++h)
        if (W == 1 || W * h + el.grp < P1) seen.see(el.su[(W * h + el.grp) * PP]);
      if (it + 1 < nit) load_l2g(it + 1);
    }
    const unsigned mx = __reduce_max_sync(lanes, seen.top());
    const int code = live && m.gexp != nullptr ? __ldg(m.gexp + e) : kFxNoGrid, ge = code >> kFxReachBits;
    const FxNorm norm{lanes, lead, smax + (it & 1) * EB + (live ? slot : 0), 2 * EB};
    if (lead) atomicMax(norm.top, mx);
    __syncthreads();
    const unsigned top = live ? *norm.top : 0u;
    const int eb = top == 0u ? 1023 : int(top >> 20);  // every value is zero: any exponent
    const bool bad = live && (code == kFxNoGrid || eb < 500 || eb > 1500);
    // the own nodes: no large value among them and not all of the Dirichlet boundary
    const bool weak = live && !bad && int(seen.top()) < fx_reach_word(top, code >> 8 & 15) &&
                      !(a.skip_dirichlet_out && dcur == (1u << (W == 1 ? P1 : (P1 - el.grp + W - 1) / W)) - 1u);
    if (el.t == 0 && el.grp == 0 && live) smax[(~it & 1) * EB + slot] = smax[(2 + (~it & 1)) * EB + slot] = 0u;
    double* wl = a.wl + size_t(e) * P3 * NC + size_t(el.t) * NC + c;
    double acc = 0.0;
    auto finish = [&](int h, int k, double w) {
      const double u = el.su[k * PP];
      if constexpr (HELM) w += a.beta * __ldg(a.Mq + e * P3 + k * PP + el.t) * u;  // Eq. (17)
      if (store) {
        if (!(a.skip_dirichlet_out && ((dcur >> h) & 1u))) wl[size_t(k) * PP * NC] = w;
        acc += w * u;
      }
    };
    bool ahead = live && it + 1 < nit;
    auto mid = [&]() {  // once, also if the element changes to FP64
      if (ahead) {
        ahead = false;
        if (Sh::NU == 2) fetch_u(it + 1);
        if (NC == 1 || (it + 1) % NC == 0) prefetch_G(elem_of(it + 1));
      }
    };
    if (live) {
      int2* A = static_cast<int2*>(el.A) + el.tj * S + el.ti;
#pragma unroll
      for (int h = 0; h < KC; ++h)
        if (const int k = W * h + el.grp; W == 1 || k < P1) A[k * PS] = fx_from_double(el.su[k * PP], eb);
    }
    bool f64 = __syncthreads_or(bad);
    if (!f64) {
      if (weak) {  // its nodes one by one
        const double* se = el.su - el.t;
        const int slack = fx_slack(a.state, c);
        bool off = false;
        if (!fx_line_reaches<P1>(el.su, PP, fx_reach_word(top, code >> 8 & 15, slack)))
#pragma unroll 1
          for (int h = 0; h < KC; ++h) {
            const int k = W * h + el.grp;
            if ((W > 1 && k >= P1) || (a.skip_dirichlet_out && ((dcur >> h) & 1u))) continue;
            off |= !fx_line_reaches<P1>(se + k * PP + el.tj * P1, 1, fx_reach_word(top, code & 15, slack)) &&
                   !fx_line_reaches<P1>(se + k * PP + el.ti, P1, fx_reach_word(top, code >> 4 & 15, slack));
          }
        if (off)
          for (int s = 0; s < EB; ++s) atomicMax(smax + (2 + (it & 1)) * EB + s, kFxUneven);
      }
      const int4* G = m.Gfx + e * 3 * P3 + el.t;
      double sc = 0.0;
      f64 = !fx_co_stages<P1, W, FxArith>(
          el, tab.D, tab.DT, live, norm,
          [&](int k, int2 r, int2 s, int2 t, long long& fr, long long& fs, long long& ft) {
            const int4 g0 = __ldcs(G + (3 * k + 0) * PP), g1 = __ldcs(G + (3 * k + 1) * PP),
                       g2 = __ldcs(G + (3 * k + 2) * PP);
            const int2 g00 = make_int2(g0.x, g0.y), g01 = make_int2(g0.z, g0.w), g02 = make_int2(g1.x, g1.y),
                       g11 = make_int2(g1.z, g1.w), g12 = make_int2(g2.x, g2.y), g22 = make_int2(g2.z, g2.w);
            fr = fx_dot3(g00, r, g01, s, g02, t);
            fs = fx_dot3(g01, r, g11, s, g12, t);
            ft = fx_dot3(g02, r, g12, s, g22, t);
          },
          mid,
          [&](int shift) { sc = wij * __hiloint2double((eb + ge - shift - (1082 - 1023)) << 20, 0); },
          [&](int h, int k, long long r, long long s, long long t) {
            finish(h, k, __ll2double_rn(r + s + t) * (tab.w[k] * sc));
          });
    }
    if (f64) {
      if (live) {
        double* A = static_cast<double*>(el.A) + el.tj * S + el.ti;
#pragma unroll
        for (int h = 0; h < KC; ++h)
          if (const int k = W * h + el.grp; W == 1 || k < P1) A[k * PS] = el.su[k * PP];
      }
      __syncthreads();
      const double* G = a.G + e * 6 * P3 + el.t;
      fx_co_stages<P1, W, F64Arith>(
          el, tab.D64, tab.DT64, live, norm,
          [&](int k, double r, double s, double t, double& fr, double& fs, double& ft) {
            const double* Gk = G + k * PP;
            const double g00 = __ldcs(Gk), g01 = __ldcs(Gk + P3), g02 = __ldcs(Gk + 2 * P3), g11 = __ldcs(Gk + 3 * P3),
                         g12 = __ldcs(Gk + 4 * P3), g22 = __ldcs(Gk + 5 * P3);
            fr = g00 * r + g01 * s + g02 * t;
            fs = g01 * r + g11 * s + g12 * t;
            ft = g02 * r + g12 * s + g22 * t;
          },
          mid, [](int) {}, [&](int h, int k, double r, double s, double t) { finish(h, k, r + s + t); });
    }
    if (Sh::NU == 1 && live && it + 1 < nit) fetch_u(it + 1);  // the own column's values were read last above
#pragma unroll
    for (int q = 0; q < NC; ++q)
      if (q == c) dot[q] += acc;
  }

  if (a.partials != nullptr) cg_alpha<NC>(dot, a.partials, a.state, red);
}

template <int P1>
FxCoTab<P1> elem_fx_tab(const DeviceMesh& m) {
  FxCoTab<P1> t;
  const FxTables& f = *m.fx;
  std::memcpy(&t.D, f.D.data(), sizeof(t.D));
  std::memcpy(&t.DT, f.DT.data(), sizeof(t.DT));
  std::memcpy(&t.D64, f.D64.data(), sizeof(t.D64));
  std::memcpy(&t.DT64, f.DT64.data(), sizeof(t.DT64));
  std::memcpy(t.w, f.w.data(), sizeof(t.w));
  return t;
}

// Blocks resident on the GPU (0: the kernel does not fit), found once per instantiation; the
// attribute that lets it use its shared memory is set on the way.
template <int P1, int NC, bool HELM, int W = 1>
int elem_fx_resident() {
  using Sh = FxCoShape<P1, W>;
  static const int n = fx_resident(reinterpret_cast<const void*>(elem_fx_kernel<P1, NC, HELM, W>), Sh::NT, Sh::SMEM);
  return n;
}

// Three threads per column while every element has an SM to itself: the launch then lasts as long as one
// element does (CG iteration in us, one / three threads: N = 4, E = 64 19.8 / 17.7; N = 5, E = 150 22.5 / 18.0;
// N = 7, E = 150 22.2 / 19.4; N = 11, E = 64 32.4 / 28.0). With several elements on an SM the warps of one
// fill the gaps of another and the extra barriers cost (N = 7: E = 256 23.5 / 22.3, 512 28.9 / 31.1, 1728
// 52 / 60; N = 9, E = 256 33.9 / 37.2). Orders 1 and 2 have too little in a line (N = 1, E = 64 14.6 / 15.4).
template <int P1, int NC>
bool elem_fx_wide(int64_t nelem) {
  return NC == 1 && P1 >= 4 && nelem <= fx_sms();
}

// Elements in a slot's sequence: one wave of resident blocks covers the mesh.
template <int P1, int NC>
int elem_fx_seq(int64_t nelem) {
  return fx_seq(nelem, FxCoShape<P1>::EB, elem_fx_resident<P1, NC, false>());
}

template <int P1, int NC>
int elem_fx_blocks_t(int64_t nelem) {
  if (elem_fx_wide<P1, NC>(nelem)) return int(nelem);  // one element per block
  const int64_t per = int64_t(FxCoShape<P1>::EB) * elem_fx_seq<P1, NC>(nelem);
  return int((nelem + per - 1) / per);
}

template <int P1, int NC, bool HELM, int W>
cudaError_t launch_elem_fx_w(const DeviceMesh& m, const ElemArgs& a, int ns, cudaStream_t s) {
  using Sh = FxCoShape<P1, W>;
  if (elem_fx_resident<P1, NC, HELM, W>() < 1) return cudaErrorInvalidConfiguration;
  elem_fx_kernel<P1, NC, HELM, W>
      <<<elem_fx_blocks_t<P1, NC>(m.nelem), Sh::NT, Sh::SMEM, s>>>(m, a, elem_fx_tab<P1>(m), ns);
  return cudaGetLastError();
}

template <int P1, int NC, bool HELM>
cudaError_t launch_elem_fx_h(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s) {
  if constexpr (NC == 1 && P1 >= 4)
    if (elem_fx_wide<P1, NC>(m.nelem)) return launch_elem_fx_w<P1, NC, HELM, 3>(m, a, 1, s);
  return launch_elem_fx_w<P1, NC, HELM, 1>(m, a, elem_fx_seq<P1, NC>(m.nelem), s);
}

template <int P1>
cudaError_t launch_elem_fx_t(const DeviceMesh& m, const ElemArgs& a, cudaStream_t s) {
  if (m.ncomp == 3) return a.beta != 0.0 ? launch_elem_fx_h<P1, 3, true>(m, a, s) : launch_elem_fx_h<P1, 3, false>(m, a, s);
  return a.beta != 0.0 ? launch_elem_fx_h<P1, 1, true>(m, a, s) : launch_elem_fx_h<P1, 1, false>(m, a, s);
}

}  // namespace ceedbp
