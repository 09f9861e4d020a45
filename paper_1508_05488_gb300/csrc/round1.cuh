// round1.cuh -- the per-point pieces of round 1 (Sec. 2.1 steps 1-3) shared by
// the streaming kernels (k_round1.cu) and the whole-set kernel (k_set.cu):
// keys and views of a point, the lexicographic extremes, the FP32 edge filter
// and the exact region tests.
#pragma once
#include "cch_internal.cuh"

namespace cch {

template <int DT>
struct PointT;
template <>
struct PointT<DT_F64> { using T = double2; };
template <>
struct PointT<DT_I32> { using T = int2; };
template <>
struct PointT<DT_F32> { using T = double2; };   // widened

// Bytes a point takes in the input (float32: one word in each vector).
template <int DT>
constexpr int in_bytes() { return DT == DT_F64 ? 16 : 8; }

// ------------------------------------------------------------- keys

// Top word of 2^-126, read as FP32: a coordinate whose top word reads below
// it in magnitude is zero or below 2^-126 in magnitude, and gets the exact
// bookkeeping -- the lower end of the domain check (nonzero magnitudes below
// 2^-400 are out of range) and the smallest top-word magnitude of the set,
// zeros included, which tells a2 whether its short FP32 view is valid.
constexpr uint32_t kTinyTopBits = (1023u - 126u) << 20;
#define kTinyTopF __uint_as_float(kTinyTopBits)

// Order-preserving key of a float64 as 32-bit words (-0.0 -> +0.0).  Also
// folds the magnitude of a nonzero value into `amin` (top word), for the
// lower end of the domain check.
__device__ __forceinline__ void f64_key_words(uint64_t b, uint32_t& kh, uint32_t& kl, uint32_t& amin) {
  uint32_t h = (uint32_t)(b >> 32), l = (uint32_t)b;
  uint32_t a = h & 0x7FFFFFFFu;
  bool nz = (a | l) != 0;
  amin = min(amin, nz ? a : 0x7FFFFFFFu);
  h = nz ? h : 0u;
  uint32_t m = (uint32_t)((int32_t)h >> 31);
  kh = h ^ (m | 0x80000000u);
  kl = l ^ m;
}

// Top key word only (no domain bookkeeping).
__device__ __forceinline__ uint32_t f64_key_hi(uint64_t b) {
  uint32_t h = (uint32_t)(b >> 32), l = (uint32_t)b;
  if (((h & 0x7FFFFFFFu) | l) == 0) h = 0;
  return h ^ ((uint32_t)((int32_t)h >> 31) | 0x80000000u);
}

__device__ __forceinline__ uint64_t kw(uint32_t h, uint32_t l) { return ((uint64_t)h << 32) | l; }

// ------------------------------------------------------------------ a1

// Lexicographic minimum over (k1, k2, idx).  All four extremes are minima:
// E1 (kx, ky), E2 (ky, kx), E3 (~kx, ~ky), E4 (~ky, ~kx); int32 packs both
// 32-bit keys into k1.
struct Lex {
  uint64_t k1, k2;
  uint32_t idx;
};

__device__ __forceinline__ bool lex_less(const Lex& a, const Lex& b) {
  return a.k1 < b.k1 || (a.k1 == b.k1 && (a.k2 < b.k2 || (a.k2 == b.k2 && a.idx < b.idx)));
}
__device__ __forceinline__ void lex_min_into(Lex& a, const Lex& b) {
  if (lex_less(b, a)) a = b;
}
// Warp-wide minima in every lane, one warp reduction (redux) per 32-bit
// word: a 64-bit minimum takes its high word's minimum, then the low words'
// minimum over the lanes that hold it; the lexicographic minimum of
// (k1, k2, idx) goes word by word the same way.
__device__ __forceinline__ uint64_t u64_warp_min(uint64_t v) {
  const uint32_t hi = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)(v >> 32));
  const uint32_t lo = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0xFFFFFFFFu);
  return kw(hi, lo);
}
__device__ __forceinline__ Lex lex_warp_min(const Lex& v) {
  const uint32_t w0 = (uint32_t)(v.k1 >> 32), w1 = (uint32_t)v.k1, w2 = (uint32_t)(v.k2 >> 32), w3 = (uint32_t)v.k2;
  const uint32_t m0 = __reduce_min_sync(0xFFFFFFFFu, w0);
  bool t = w0 == m0;
  const uint32_t m1 = __reduce_min_sync(0xFFFFFFFFu, t ? w1 : 0xFFFFFFFFu);
  t = t && w1 == m1;
  const uint32_t m2 = __reduce_min_sync(0xFFFFFFFFu, t ? w2 : 0xFFFFFFFFu);
  t = t && w2 == m2;
  const uint32_t m3 = __reduce_min_sync(0xFFFFFFFFu, t ? w3 : 0xFFFFFFFFu);
  t = t && w3 == m3;
  Lex r;
  r.k1 = kw(m0, m1);
  r.k2 = kw(m2, m3);
  r.idx = __reduce_min_sync(0xFFFFFFFFu, t ? v.idx : 0xFFFFFFFFu);
  return r;
}

template <int DT>
__device__ __forceinline__ void cand_keys(uint32_t xh, uint32_t xl, uint32_t yh, uint32_t yl, int e,
                                          uint64_t& k1, uint64_t& k2) {
  if constexpr (DT == DT_F64) {
    uint64_t kx = kw(xh, xl), ky = kw(yh, yl);
    switch (e) {
      case 0: k1 = kx; k2 = ky; break;
      case 1: k1 = ky; k2 = kx; break;
      case 2: k1 = ~kx; k2 = ~ky; break;
      default: k1 = ~ky; k2 = ~kx; break;
    }
  } else {
    switch (e) {
      case 0: k1 = kw(xh, yh); break;
      case 1: k1 = kw(yh, xh); break;
      case 2: k1 = kw(~xh, ~yh); break;
      default: k1 = kw(~yh, ~xh); break;
    }
    k2 = 0;
  }
}

// Key words of one point (int32: one word per coordinate, low words 0).
template <int DT>
__device__ __forceinline__ void a1_words(const typename PointT<DT>::T& p, uint32_t& xh, uint32_t& xl,
                                         uint32_t& yh, uint32_t& yl, uint32_t& amin) {
  if constexpr (DT == DT_F64) {
    f64_key_words((uint64_t)__double_as_longlong(p.x), xh, xl, amin);
    f64_key_words((uint64_t)__double_as_longlong(p.y), yh, yl, amin);
  } else {
    xh = (uint32_t)p.x ^ 0x80000000u;
    yh = (uint32_t)p.y ^ 0x80000000u;
    xl = yl = 0;
  }
}

// Whether a point can improve any of the four running minima: only the top
// 32 bits of each k1 are compared here; the full comparison runs in
// a1_update, which is rare (new minima, or ties of the top words).
__device__ __forceinline__ bool a1_maybe(uint32_t xh, uint32_t yh, const uint32_t th[4]) {
  return xh <= th[0] || yh <= th[1] || ~xh <= th[2] || ~yh <= th[3];
}

// Full update (indices grow within a thread: a strict order keeps the
// smallest index among equal keys).
template <int DT>
__device__ __forceinline__ void a1_update(uint32_t xh, uint32_t xl, uint32_t yh, uint32_t yl, uint32_t i,
                                          Lex best[4]) {
#pragma unroll
  for (int e = 0; e < 4; e++) {
    Lex c;
    cand_keys<DT>(xh, xl, yh, yl, e, c.k1, c.k2);
    if (c.k1 < best[e].k1 || (c.k1 == best[e].k1 && c.k2 < best[e].k2)) {
      best[e].k1 = c.k1;
      best[e].k2 = c.k2;
      best[e].idx = i;
    }
  }
}

// Thresholds shared by the warp: the smallest top word of each running
// minimum over the lanes.  A point whose top word exceeds the warp's cannot
// be the set's extreme, so only points at or below it take the full update;
// sharing the bound across the warp keeps that rare.
__device__ __forceinline__ void a1_thresholds(const Lex best[4], uint32_t th[4]) {
#pragma unroll
  for (int e = 0; e < 4; e++) th[e] = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)(best[e].k1 >> 32));
}

// float64 filter on the top 32 bits of each coordinate read as an FP32
// number.  That reading is non-decreasing in the coordinate wherever it is
// not NaN and -0.0 and +0.0 compare equal; the largest magnitudes (from
// 2^1017 on) and Inf / NaN inputs read as +-Inf, ordered beyond every other
// reading, or as NaN, which the unordered tests below let through -- either
// way such a value reaches the exact update, becomes an extreme, and
// setup_set reports it.  A threshold is the top word of the warp's running bound
// turned back from key to bits: a point passes when its top word is at or
// beyond the bound's, so the exact keys still decide every tie.
__device__ __forceinline__ float a1_bound_f(uint32_t keyhi) {
  const uint32_t raw = (keyhi & 0x80000000u) ? (keyhi ^ 0x80000000u) : ~keyhi;
  return __uint_as_float(raw);
}
__device__ __forceinline__ void a1_thresholds_f(const Lex best[4], float thf[4]) {
#pragma unroll
  for (int e = 0; e < 4; e++) {
    const uint32_t t = __reduce_min_sync(0xFFFFFFFFu, (uint32_t)(best[e].k1 >> 32));
    thf[e] = a1_bound_f(e >= 2 ? ~t : t);
  }
}

// Bucket of the stairs map: monotone non-decreasing in u.
__device__ __forceinline__ int stair_bucket(float u, float lo, float scale) {
  float t = __fmul_rn(__fsub_rn(u, lo), scale);
  int b = __float2int_rd(t);
  return min(max(b, 0), kStairB - 1);
}

// Order-preserving unsigned key of a (non-NaN) float.
__device__ __forceinline__ uint32_t f32_order(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// FP32 view of a point used by the filter and the stairs (truncated float64,
// rounded int32): monotone in each coordinate.  A float32 input is its own
// view (view_at reads it from the vectors).
template <int DT>
__device__ __forceinline__ void f32_view(const typename PointT<DT>::T& p, float& X, float& Y) {
  static_assert(DT != DT_F32, "float32 views come from view_at");
  if constexpr (DT == DT_F64) {
    X = f64_trunc_f32((uint64_t)__double_as_longlong(p.x));
    Y = f64_trunc_f32((uint64_t)__double_as_longlong(p.y));
  } else {
    X = __int2float_rn(p.x);
    Y = __int2float_rn(p.y);
  }
}

// FP32 view of input point i (set offset included).
template <int DT>
__device__ __forceinline__ void view_at(const Job& j, int64_t i, float& X, float& Y) {
  if constexpr (DT == DT_F32) {
    X = reinterpret_cast<const float*>(j.pts)[i];
    Y = j.ys[i];
  } else {
    f32_view<DT>(input_point<typename PointT<DT>::T>(j, i), X, Y);
  }
}

// The same FP32 view in three integer operations per coordinate, for sets
// whose coordinates all have magnitude in [2^-126, 2^60] (SF_SHORTVIEW): the
// exponent is rebiased on the signed top word (no borrow reaches the sign:
// the magnitude's top word is at least 0x38100000) and shifted with the three
// leading bits of the low word; the bits equal f64_trunc_f32's.
__device__ __forceinline__ float f64_view_short(uint64_t b) {
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  const uint32_t t = hi - 0x38000000u;
  return __uint_as_float(__funnelshift_l(lo, t, 3) | (hi & 0x80000000u));
}
template <int DT, bool SHORT>
__device__ __forceinline__ void f32_view_a2(const typename PointT<DT>::T& p, float& X, float& Y) {
  if constexpr (DT == DT_F64 && SHORT) {
    X = f64_view_short((uint64_t)__double_as_longlong(p.x));
    Y = f64_view_short((uint64_t)__double_as_longlong(p.y));
  } else {
    f32_view<DT>(p, X, Y);
  }
}

// Compared coordinate of region r (0..3) as the order word of its FP32 view
// in "smaller is better" form: R1 y, R2 -x, R3 -y, R4 x (-0.0 read as +0.0).
// The view is non-decreasing in the coordinate, so a strictly larger word
// means a strictly worse coordinate: the dominance tables hold these words.
__device__ __forceinline__ uint32_t cmp_view_order(float X, float Y, int r) {
  const float v = (r & 1) ? X : Y;
  return f32_order(__fadd_rn((r == 1 || r == 2) ? -v : v, 0.0f));
}

// Sort coordinate (FP32 view) of region r: R1 x asc, R2 y asc, R3 x desc, R4 y desc.
__device__ __forceinline__ float sort_u(float X, float Y, int r) {
  switch (r) {
    case 0: return X;
    case 1: return Y;
    case 2: return -X;
    default: return -Y;
  }
}

// FP32 filter of the directed edge a -> b (see setup_set): coefficients of
// orient(a, b, p) = A py - B px + C and the bound E on its FP32 evaluation
// error; a degenerate edge (a = b) is always "inside", without the filter
// (filt false) nothing is.
static __device__ void edge_filter(double ax, double ay, double bx, double by, double xm, double ym, bool filt,
                            float& fA, float& fB, float& fC, float& fE) {
  const double u = 5.9604644775390625e-08;
  if (!filt) {
    fA = 0.f; fB = 0.f; fC = 0.f; fE = __int_as_float(0x7F800000);
  } else if (ax == bx && ay == by) {
    fA = 0.f; fB = 0.f; fC = 1.f; fE = 0.f;
  } else {
    double A = bx - ax, B = by - ay;
    double C = B * ax - A * ay;
    double Mc = fabs(B) * fabs(ax) + fabs(A) * fabs(ay);
    double E = 6.0 * u * (fabs(A) * ym + fabs(B) * xm + Mc)
             + (fabs(A) + fabs(B)) * 2.350988701644575e-38      // 2^-125
             + 3.5032461608120427e-45 * (xm + ym + 1.0);        // 2^-147
    fA = __double2float_rn(A);
    fB = __double2float_rn(B);
    fC = __double2float_rn(C);
    fE = __double2float_ru(E);
  }
}

// Minimum / maximum that return NaN when either operand is NaN, so that a
// NaN coordinate shows up in a lane's running extremes.
__device__ __forceinline__ float fmin_nan(float a, float b) {
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float fmax_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}

// Exact region test of one point (every edge: FP64 filter, then expansion
// arithmetic).  Kept out of line: only points the FP32 filter cannot decide
// get here.
static __device__ __noinline__ int region_exact_f64(double px, double py, const double* ex, const double* ey,
                                             uint32_t flags) {
  for (int k = 0; k < 4; k++) {
    if (flags & (SF_DEGEN0 << k)) continue;
    int k1 = (k + 1) & 3;
    if (orient_f64(ex[k], ey[k], ex[k1], ey[k1], px, py) < 0) return k + 1;
  }
  return 0;
}

static __device__ __noinline__ int region_exact_i32_wide(int px, int py, const double* ex, const double* ey,
                                                  uint32_t flags) {
  for (int k = 0; k < 4; k++) {
    if (flags & (SF_DEGEN0 << k)) continue;
    int k1 = (k + 1) & 3;
    if (orient_i32((int)ex[k], (int)ey[k], (int)ex[k1], (int)ey[k1], px, py, true) < 0) return k + 1;
  }
  return 0;
}

// The same with 64-bit products where the set's spans allow them.
static __device__ __noinline__ int region_exact_i32(int px, int py, const double* ex, const double* ey,
                                                    uint32_t flags) {
  if (flags & SF_WIDE) return region_exact_i32_wide(px, py, ex, ey, flags);
  for (int k = 0; k < 4; k++) {
    if (flags & (SF_DEGEN0 << k)) continue;
    const int k1 = (k + 1) & 3;
    if (orient_i32((int)ex[k], (int)ey[k], (int)ex[k1], (int)ey[k1], px, py, false) < 0) return k + 1;
  }
  return 0;
}

}  // namespace cch
