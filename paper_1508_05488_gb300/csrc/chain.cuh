// chain.cuh -- pieces of the chain hull (Sec. 2.1 steps 6-7) shared by
// k_chain.cu and the whole-set kernel (k_set.cu): orientation of chain points
// and the bridge walk that joins two adjacent convex chains.
#pragma once
#include "cch_internal.cuh"

namespace cch {

template <int DT>
struct PT;
template <>
struct PT<DT_F64> { using T = double2; };
template <>
struct PT<DT_I32> { using T = int2; };

template <int DT>
__device__ __forceinline__ bool same_pt(const typename PT<DT>::T& a, const typename PT<DT>::T& b) {
  return a.x == b.x && a.y == b.y;   // value equality: -0.0 == +0.0
}

// Merge two adjacent convex chains given by (head, tail) into the left one.
// Links, flags, points and orientation go through the accessor (shared or
// global memory).
template <class A>
__device__ void merge_chains(A& acc, int& hl, int& tl, int hr, int tr) {
  if (hr < 0) return;
  if (hl < 0) { hl = hr; tl = tr; return; }
  int a = tl, b = hr;
  for (;;) {
    bool moved = false;
    while (a != hl && acc.orient(acc.prv(a), a, b) <= 0) {
      acc.kill(a);
      a = acc.prv(a);
      moved = true;
    }
    while (b != tr && acc.orient(a, b, acc.nxt(b)) <= 0) {
      acc.kill(b);
      b = acc.nxt(b);
      moved = true;
    }
    if (!moved) break;
  }
  acc.link(a, b);
  tl = tr;
}

// Orientation of three chain points: float64 through the FP32 filter on
// their views (when the set's coordinates allow), then exactly; int32
// exactly in 64/128-bit integers.
template <int DT>
__device__ __forceinline__ int orient_chain(const typename PT<DT>::T& a, const typename PT<DT>::T& b,
                                            const typename PT<DT>::T& c, float4 A, float4 B, float4 C,
                                            bool flag) {
  if constexpr (DT == DT_F64) return orient_f64_split(a, b, c, A, B, C, flag);
  else return orient_i32(a.x, a.y, b.x, b.y, c.x, c.y, flag);
}

constexpr int kPeelRounds = 48;   // peeling rounds before the stack-and-merge fallback

}  // namespace cch
