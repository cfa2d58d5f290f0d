// The direct-stiffness sum Q^T of one or more nodes per thread: w[g] = sum of the node's local values in
// slot order (deterministic, no atomics), with the loads of all nodes in flight together.
//
// head[g] (built at setup) takes a node to its values without going through the CSR offsets: an element
// interior's only slot itself, or the place of a list in `slots` whose last entry carries bit 31. A node
// with one slot is then two dependent loads away from its value instead of three, one with up to four
// slots three loads away instead of four to six.
#pragma once

#include "common.cuh"
#include "df.cuh"

namespace ceedbp {

constexpr int kHeadDirichlet = -1;              // also nodes past the end
constexpr int kHeadEmpty = int(0x80000000u);    // a node that no element touches
constexpr int kSlotMask = 0x7fffffff;
// U, the nodes a thread has in flight: with three components one, whose registers leave room for more blocks
// (FP64 update, N = 7, 12^3 elements: 43 us, 51 with two); with one component two, unless the grid holds all
// nodes already, when a second one only costs registers (N = 7: 257 us with two, 371 with one at 2^16 elements,
// 18.7 and 14.7 us at 8^3)
inline bool gather_one(int64_t n, int blocks) { return n <= int64_t(blocks) * 256; }

__device__ __forceinline__ void gather_add(double& w, double v) { w += v; }
__device__ __forceinline__ void gather_add(float& w, float v) { w += v; }
__device__ __forceinline__ void gather_add(dfloat& w, dfloat v) { w = dw_add(w, v); }
__device__ __forceinline__ double gather_load(const double* p) { return __ldcs(p); }
__device__ __forceinline__ float gather_load(const float* p) { return __ldcs(p); }
__device__ __forceinline__ dfloat gather_load(const dfloat* p) {
  const float2 v = __ldcs(reinterpret_cast<const float2*>(p));
  return dfloat{v.x, v.y};
}

// Nodes g0, g0 + stride, ... (U of them): hd[h] their heads (kHeadDirichlet: nothing to do), w[h] their sums.
template <int U, int NC, class T>
__device__ __forceinline__ void gather_nodes(const int* __restrict__ head, const int* __restrict__ slots,
                                             const T* __restrict__ wl, int64_t g0, int64_t stride, int64_t n,
                                             int (&hd)[U], T (&w)[U][NC]) {
#pragma unroll
  for (int h = 0; h < U; ++h) hd[h] = g0 + h * stride < n ? __ldg(head + g0 + h * stride) : kHeadDirichlet;
  int sl[U][4];
#pragma unroll
  for (int h = 0; h < U; ++h) {
    const int o = hd[h] < kHeadDirichlet && hd[h] != kHeadEmpty ? -hd[h] - 2 : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) sl[h][k] = __ldg(slots + o + k);
    if (hd[h] >= 0) sl[h][0] = hd[h] | ~kSlotMask;  // one slot, the last
  }
  T v[U][4][NC];
#pragma unroll
  for (int h = 0; h < U; ++h) {
    bool on = hd[h] != kHeadDirichlet && hd[h] != kHeadEmpty;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        v[h][k][c] = T{};
        if (on) v[h][k][c] = gather_load(wl + size_t(sl[h][k] & kSlotMask) * NC + c);
      }
      on = on && sl[h][k] >= 0;  // the last entry has bit 31 set
    }
  }
#pragma unroll
  for (int h = 0; h < U; ++h) {
    bool on = hd[h] != kHeadDirichlet && hd[h] != kHeadEmpty;
#pragma unroll
    for (int c = 0; c < NC; ++c) w[h][c] = v[h][0][c];
#pragma unroll
    for (int k = 1; k < 4; ++k) {
      on = on && sl[h][k - 1] >= 0;
      if (on) {
#pragma unroll
        for (int c = 0; c < NC; ++c) gather_add(w[h][c], v[h][k][c]);
      }
    }
    on = on && sl[h][3] >= 0;
    if (on) {  // more than four slots: the rest four at a time
      const int* s = slots + (-hd[h] - 2) + 4;
      bool more = true;
      while (more) {
        int q[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) q[k] = __ldg(s + k);
        T y[4][NC];
        bool in = true;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            y[k][c] = T{};
            if (in) y[k][c] = gather_load(wl + size_t(q[k] & kSlotMask) * NC + c);
          }
          in = in && q[k] >= 0;
        }
        more = in;
        in = true;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (in) {
#pragma unroll
            for (int c = 0; c < NC; ++c) gather_add(w[h][c], y[k][c]);
          }
          in = in && q[k] >= 0;
        }
        s += 4;
      }
    }
  }
}

}  // namespace ceedbp
