// k_sieve.cu -- one streaming pass for large sets: a point well inside the
// convex hull of a sample is no hull vertex, so the set's hull is that of the
// points the sample's polygon does not cover.
//
// The pipeline of k_round1.cu reads every point twice (the extremes fix the
// regions before the classification) and its dominance tables leave many
// points where the hull is round (20M disk: 60,000).  Here
//   k_table    one cluster per set reduces a spread sample to a polygon and
//              writes tables of bands, of Y with the polygon's left and right
//              chord in each and of X with its lower and upper one;
//   k_sieve    reads every point once and lists the indices of those that
//              neither axis' chords certainly hold, in index order;
//   k_refine   one cluster per set gathers the listed points; where they are
//              many it builds the polygon of the listed points themselves and
//              lists only those outside it;
//   k_set      (k_set.cu) runs the method (Sec. 2.1) on the listed points.
// A batch's sets above kSetMax points go the same way, every set with a table
// of its own (one CTA) and without k_refine.
// Sets whose points mostly lie on or beside their hull (the sample tells) take
// the pipeline, which k_refine's flag lets the later launches know.
//
// Why the hull is unchanged.  A dropped point p lies strictly inside the
// convex hull of input points, so it is neither a strict vertex nor equal to
// one; the listed points therefore have the same strict hull, and being listed
// in index order they have the same smallest index per vertex.  Coordinates
// that fail the float64 domain check are always listed, so the check reports
// the same status.
//
// The bands (of Y; those of X are the same with the axes exchanged, and hold
// where the polygon runs level).  Everything is computed on FP32 views (float64 truncated, int32
// rounded: within 2 u |v| of v, u = 2^-24; magnitudes below 2^-126 within
// 2^-126, covered because the maxima xm, ym of |X|, |Y| over the sample are at
// least 2^-100).  The sample's left and right polylines run from its lowest to
// its highest point through the leftmost (rightmost) sample point of every
// band, peeled towards convexity; convexity is never relied on, every point of
// a polyline is in the hull.  Band b covers the Y with s Y + o in [b, b + 1);
// rounding moves that border by less than d = 2^-20 ym.  Its left chord joins
// the left polyline's points at the band's borders moved out by d, so both
// ends are within 2 u (xm, ym) plus the interpolation's 9 u xm of points of the
// hull, and with the right chord they span a trapezoid inside it (up to that).
// X > m Y + a + E with E = 64 u (xm + |m| ym) bounds those errors, the
// rounding of m, a (11 u xm + 4 u |m| ym) and of the test, and the view's
// distance from the point: p is strictly right of the left chord of the exact
// points; the right chord likewise.
#include <algorithm>
#include <cooperative_groups.h>

#include "cch_internal.cuh"
#include "round1.cuh"

namespace cch {
namespace cg = cooperative_groups;

namespace {

constexpr int kTabThreads = 1024;                   // of k_refine, and of k_table on a single set
constexpr int kTabBatchThreads = 256;               // of k_table on a batch's sets: 4096 sample points each, four
                                                    // sets per SM (512 threads, two: 37 us for 409 sets, 30
                                                    // so; 1024 where every set has an SM to itself: 5 to 8
                                                    // us less a call)
constexpr int kTabItems = 8, kTabBatchItems = 16;   // points per thread at most
constexpr int kPeel = 40;                           // peeling rounds at most
constexpr int64_t kLeast = 8;                       // where more than this share of a set is left, little of it
                                                    // lies inside even its own polygon (k_refine)
constexpr int64_t kSvMost = 131072;                 // points that k_refine takes
constexpr uint32_t kPlain = 2048;                   // lists up to this size go to k_set as they are

template <int DT>
using RawPt = typename std::conditional<DT == DT_F64, uint4, uint2>::type;   // a point's words

// View of a point; false where the point takes no part in a polygon and is
// never dropped (outside the float64 domain, or beyond 2^60 where the views
// end; float32 NaN).
template <int DT>
__device__ __forceinline__ bool sieve_view_of(const RawPt<DT>& p, float& X, float& Y) {
  if constexpr (DT == DT_F64) {
    const uint64_t bx = ((uint64_t)p.y << 32) | p.x, by = ((uint64_t)p.w << 32) | p.z;
    X = f64_trunc_f32(bx);
    Y = f64_trunc_f32(by);
    return max(p.y & 0x7FFFFFFFu, p.w & 0x7FFFFFFFu) < ((1023u + 60u) << 20) && !f64_bad(bx) && !f64_bad(by);
  } else if constexpr (DT == DT_F32) {
    X = __uint_as_float(p.x);
    Y = __uint_as_float(p.y);
    return fabsf(X) < 1152921504606846976.0f && fabsf(Y) < 1152921504606846976.0f;
  } else {
    X = __int2float_rn((int)p.x);
    Y = __int2float_rn((int)p.y);
    return true;
  }
}
template <int DT>
__device__ __forceinline__ bool sieve_view(const Job& j, int64_t i, float& X, float& Y) {
  if constexpr (DT == DT_F32)
    return sieve_view_of<DT>(make_uint2(reinterpret_cast<const uint32_t*>(j.pts)[i], __float_as_uint(j.ys[i])), X, Y);
  else
    return sieve_view_of<DT>(reinterpret_cast<const RawPt<DT>*>(j.pts)[i], X, Y);
}

// The band map and chords of one axis: band of u is s u + o, dropped is what
// lies strictly between the chords lo + ml u and hi + mh u in the other.
// G: the table is global memory that this kernel writes (not from L1).
template <int R, bool G>
__device__ __forceinline__ bool sieve_between(const float4* tab, float s, float o, float u, float v) {
  const uint32_t b = min(__float2uint_rz(__fmaf_rn(u, s, o)), (uint32_t)(R + 1));   // NaN, negative: 0
  const float4 c = G ? __ldcg(tab + b) : tab[b];
  return v > __fmaf_rn(c.y, u, c.x) && v < __fmaf_rn(c.w, u, c.z);
}
// Certainly inside: by the bands of Y, else by those of X.
template <int R, bool G>
__device__ __forceinline__ bool sieve_inside(const float4* tab, const SieveHdr& h, float X, float Y) {
  return sieve_between<R, G>(tab, h.s[0], h.o[0], Y, X) || sieve_between<R, G>(tab + R + 2, h.s[1], h.o[1], X, Y);
}

// Sides: 0 left, 1 right (bands u = Y, compared v = X, -X), 2 bottom, 3 top
// (u = X, v = Y, -Y).  A polyline point is (v, u).
template <int R, int T>
struct TabSmem {
  static constexpr int W = T / 32;
  uint2 bv[2][R];               // per axis and band: order words of the smallest v of its two sides
  uint2 bu[2][R];               // bits of those points' u
  float2 pl[4][2][R + 2];       // polylines, ping-pong
  uint64_t ext[W][4];
  uint64_t gext[4];             // this CTA's extremes, read by the cluster
  uint32_t w32[4][2][W / 4];
  uint32_t plen[4], pbuf[4];    // the polylines' lengths and buffers
  uint32_t cnt;                 // leader: sample points outside; k_refine: points kept
  uint32_t pre[W];
  uint32_t upre[T == kTabThreads ? kSvMaxUnits : 1];   // k_refine: listed points before each unit
};

__device__ __forceinline__ float unorder(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k ^ 0x80000000u) : ~k);
}

template <int CL>
__device__ __forceinline__ void cl_sync() {
  if constexpr (CL > 1) cg::this_cluster().sync();
  else __syncthreads();
}
template <int CL, typename T>
__device__ __forceinline__ T* cl_map(T* p, int r) {
  if constexpr (CL > 1) return cg::this_cluster().map_shared_rank(p, r);
  else return p;
}

// Barrier of one side's quarter of the CTA.
template <int T>
__device__ __forceinline__ void side_sync(int side) {
  asm volatile("bar.sync %0, %1;" :: "r"(side + 1), "r"(T / 4) : "memory");
}

// Inclusive warp prefix sum.
__device__ __forceinline__ uint32_t warp_incl_sum(uint32_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Polygon tables of the cluster's points (NI views per thread, `valid`
// bit k: item k), by every thread of the cluster.  They go to `tab` and `hdr`
// (global memory) and are visible to the cluster on return; false where there
// are none.
template <int R, int CL, int T, int NI>
__device__ bool build_table(TabSmem<R, T>& m, const float (&X)[NI], const float (&Y)[NI], uint32_t valid,
                            int rank, float4* tab, SieveHdr* hdr) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // extremes: per side the smallest v (and the smallest u among them)
  {
    uint64_t e[4] = {~0ull, ~0ull, ~0ull, ~0ull};
#pragma unroll
    for (int k = 0; k < NI; k++) {
      if ((valid >> k) & 1u) {
        const uint32_t ox = f32_order(X[k]), oy = f32_order(Y[k]);
        e[0] = min(e[0], kw(ox, oy));
        e[1] = min(e[1], kw(~ox, oy));
        e[2] = min(e[2], kw(oy, ox));
        e[3] = min(e[3], kw(~oy, ox));
      }
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {
      e[q] = u64_warp_min(e[q]);
      if (lane == 0) m.ext[warp][q] = e[q];
    }
    for (int i = tid; i < 2 * R; i += T) (&m.bv[0][0])[i] = make_uint2(0xFFFFFFFFu, 0xFFFFFFFFu);
    __syncthreads();
    if (warp < 4) {
      const uint64_t g = u64_warp_min(lane < T / 32 ? m.ext[lane][warp] : ~0ull);
      if (lane == 0) m.gext[warp] = g;
    }
    if (tid == 0) m.cnt = 0;
  }
  cl_sync<CL>();
  uint64_t e[4];
  if constexpr (CL > 1) {
    // lane 4 c + q reads extreme q of CTAs c and c + 8
    static_assert(CL % 8 == 0, "one lane per CTA and side");
    uint64_t v = cl_map<CL>(m.gext, lane >> 2)[lane & 3];
#pragma unroll
    for (int c = 8; c < CL; c += 8) v = min(v, cl_map<CL>(m.gext, c + (lane >> 2))[lane & 3]);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) v = min(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
#pragma unroll
    for (int q = 0; q < 4; q++) e[q] = __shfl_sync(0xFFFFFFFFu, v, q);
  } else {
#pragma unroll
    for (int q = 0; q < 4; q++) e[q] = m.gext[q];
  }
  const float x0 = unorder((uint32_t)(e[0] >> 32)), x1 = unorder(~(uint32_t)(e[1] >> 32));
  const float y0 = unorder((uint32_t)(e[2] >> 32)), y1 = unorder(~(uint32_t)(e[3] >> 32));
  const float xm = fmaxf(fabsf(x0), fabsf(x1)), ym = fmaxf(fabsf(y0), fabsf(y1));
  const float least = 7.8886090522101181e-31f;       // 2^-100
  const bool ok = e[0] != ~0ull && y1 > y0 && x1 > x0 && xm >= least && ym >= least;   // the same in every thread
  const float by = __fdiv_rn((float)R, y1 - y0), bx = __fdiv_rn((float)R, x1 - x0);
  if (!ok || !(by < 1.0e36f) || !(bx < 1.0e36f)) {
    cl_sync<CL>();                                   // nobody leaves while its words are read
    return false;
  }
  // the smallest v of every band, then its u (any point that holds the minimum)
#pragma unroll
  for (int k = 0; k < NI; k++) {
    if ((valid >> k) & 1u) {
      const int b = min((int)((Y[k] - y0) * by), R - 1), c = min((int)((X[k] - x0) * bx), R - 1);
      const uint32_t ox = f32_order(X[k]), oy = f32_order(Y[k]);
      const uint2 p = m.bv[0][b], q = m.bv[1][c];
      if (ox < p.x) atomicMin(&m.bv[0][b].x, ox);
      if (~ox < p.y) atomicMin(&m.bv[0][b].y, ~ox);
      if (oy < q.x) atomicMin(&m.bv[1][c].x, oy);
      if (~oy < q.y) atomicMin(&m.bv[1][c].y, ~oy);
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NI; k++) {
    if ((valid >> k) & 1u) {
      const int b = min((int)((Y[k] - y0) * by), R - 1), c = min((int)((X[k] - x0) * bx), R - 1);
      const uint32_t ox = f32_order(X[k]), oy = f32_order(Y[k]);
      const uint2 p = m.bv[0][b], q = m.bv[1][c];
      if (ox == p.x) m.bu[0][b].x = __float_as_uint(Y[k]);
      if (~ox == p.y) m.bu[0][b].y = __float_as_uint(Y[k]);
      if (oy == q.x) m.bu[1][c].x = __float_as_uint(X[k]);
      if (~oy == q.y) m.bu[1][c].y = __float_as_uint(X[k]);
    }
  }
  cl_sync<CL>();
  if constexpr (CL > 1) {
    // each CTA merges its share of the bands into the leader's copy
    constexpr int S = 4 * R / CL;                    // words
    static_assert(S <= T, "one band word per thread");
    if (tid < S) {
      const int i = rank * S + tid;
      uint32_t w[CL], v[CL];
#pragma unroll
      for (int c = 0; c < CL; c++) {
        w[c] = cl_map<CL>(reinterpret_cast<uint32_t*>(m.bv), c)[i];
        v[c] = cl_map<CL>(reinterpret_cast<uint32_t*>(m.bu), c)[i];
      }
      uint32_t bw = w[0], bu = v[0];
#pragma unroll
      for (int c = 1; c < CL; c++)
        if (w[c] < bw) { bw = w[c]; bu = v[c]; }
      // only this thread reads or writes word i of the leader's copy now
      cl_map<CL>(reinterpret_cast<uint32_t*>(m.bv), 0)[i] = bw;
      cl_map<CL>(reinterpret_cast<uint32_t*>(m.bu), 0)[i] = bu;
    }
    cl_sync<CL>();
  }
  if (rank == 0) {
    // one side per quarter of the CTA: polyline of the band points, then peeling
    constexpr int H = T / 4, HW = H / 32, PB = (R + H - 1) / H, Q = (R + 2 + H - 1) / H;
    const int side = tid / H, t = tid - side * H, sw = t >> 5;
    float2* cur = m.pl[side][0];
    float2* nxt = m.pl[side][1];
    const float sg = (side & 1) ? -1.f : 1.f;
    const float sb = side < 2 ? by : bx;
    const uint32_t* bv = reinterpret_cast<const uint32_t*>(m.bv[side >> 1]) + (side & 1);
    const uint32_t* bu = reinterpret_cast<const uint32_t*>(m.bu[side >> 1]) + (side & 1);
    uint32_t n;
    {
      uint32_t c = 0;
#pragma unroll
      for (int q = 0; q < PB; q++) { const int b = t * PB + q; c += b < R && bv[2 * b] != 0xFFFFFFFFu; }
      const uint32_t x = warp_incl_sum(c);
      if (lane == 31) m.w32[side][0][sw] = x;
      side_sync<T>(side);
      uint32_t pre = x - c + 1, tot = 0;
#pragma unroll
      for (int q = 0; q < HW; q++) { const uint32_t v = m.w32[side][0][q]; pre += q < sw ? v : 0u; tot += v; }
#pragma unroll
      for (int q = 0; q < PB; q++) {
        const int b = t * PB + q;
        if (b < R && bv[2 * b] != 0xFFFFFFFFu) {
          const uint32_t w = bv[2 * b];
          cur[pre++] = make_float2(unorder((side & 1) ? ~w : w), __uint_as_float(bu[2 * b]));
        }
      }
      n = tot + 2;
      // the ends: the extremes of u
      const uint64_t elo = side < 2 ? e[2] : e[0], ehi = side < 2 ? e[3] : e[1];
      if (t == 0) cur[0] = make_float2(unorder((uint32_t)elo), unorder((uint32_t)(elo >> 32)));
      if (t == 1) cur[n - 1] = make_float2(unorder((uint32_t)ehi), unorder(~(uint32_t)(ehi >> 32)));
      side_sync<T>(side);
    }
    auto keeps = [&](uint32_t i) {
      if (i == 0 || i == n - 1) return true;
      const float2 a = cur[i - 1], b = cur[i], c = cur[i + 1];
      const float d = (c.x - a.x) * ((b.y - a.y) * sb) - ((c.y - a.y) * sb) * (b.x - a.x);
      return d * sg > 0.f;
    };
    int round = 0;
    bool conv = false;
    for (; round < kPeel && !conv && n > 64; round++) {
      const uint32_t per = (n + H - 1) / H, i0 = t * per;
      uint32_t keep = 0;
#pragma unroll
      for (int q = 0; q < Q; q++)
        if (q < (int)per && i0 + q < n && keeps(i0 + q)) keep |= 1u << q;
      const uint32_t c = __popc(keep), x = warp_incl_sum(c);
      uint32_t* sh = m.w32[side][(round + 1) & 1];
      if (lane == 31) sh[sw] = x;
      side_sync<T>(side);
      uint32_t pre = x - c, tot = 0;
#pragma unroll
      for (int q = 0; q < HW; q++) { const uint32_t v = sh[q]; pre += q < sw ? v : 0u; tot += v; }
      conv = tot == n;
      if (!conv) {
#pragma unroll
        for (int q = 0; q < Q; q++)
          if ((keep >> q) & 1u) nxt[pre++] = cur[i0 + q];
        float2* z = cur; cur = nxt; nxt = z;
        n = tot;
        side_sync<T>(side);
      }
    }
    // the rest by the side's first warp, without CTA barriers
    if (sw == 0) {
      for (; round < kPeel && !conv; round++) {
        uint32_t keep = 0;                             // n <= 64 here
        if (2 * lane < (int)n && keeps(2 * lane)) keep |= 1u;
        if (2 * lane + 1 < (int)n && keeps(2 * lane + 1)) keep |= 2u;
        const uint32_t c = __popc(keep), x = warp_incl_sum(c);
        const uint32_t tot = __shfl_sync(0xFFFFFFFFu, x, 31);
        uint32_t pre = x - c;
        conv = tot == n;
        if (!conv) {
          if (keep & 1u) nxt[pre++] = cur[2 * lane];
          if (keep & 2u) nxt[pre] = cur[2 * lane + 1];
          float2* z = cur; cur = nxt; nxt = z;
          n = tot;
          __syncwarp();
        }
      }
      if (lane == 0) { m.plen[side] = n; m.pbuf[side] = cur == m.pl[side][0] ? 0u : 1u; }
    }
    __syncthreads();
    // chords of both axes' bands, one thread per band
    auto at = [&](int sd, float u) {                             // the polyline's v at u, within its ends
      const float2* v = m.pl[sd][m.pbuf[sd]];
      int l = 0, h = (int)m.plen[sd] - 2;
      while (l < h) {
        const int c = (l + h + 1) >> 1;
        if (v[c].y <= u) l = c; else h = c - 1;
      }
      const float2 a = v[l], b = v[l + 1];
      const float dy = b.y - a.y;
      const float f = dy > 0.f ? fminf(fmaxf(__fdiv_rn(u - a.y, dy), 0.f), 1.f) : 0.f;
      return __fmaf_rn(f, b.x - a.x, a.x);
    };
    const float inf = __int_as_float(0x7F800000);
    for (int i = tid; i < 2 * R + 4; i += T) {
      const int ax = i < 2 * R ? i / R : i & 1;                  // the 2 R bands, then the four ends
      const int b = i < 2 * R ? i - ax * R + 1 : (i - 2 * R) / 2 * (R + 1);
      const float u0 = ax ? x0 : y0, u1 = ax ? x1 : y1, um = ax ? xm : ym, vm = ax ? ym : xm;
      const float d = um * 9.5367431640625e-07f;                 // 2^-20 um
      const float ua = u0 + 2.f * d, ub = u1 - 2.f * d;
      const float s = __fdiv_rn((float)R, ub - ua), o = __fmaf_rn(-ua, s, 1.f);
      const bool rows = ub > ua && s < 1.0e36f;
      float4 c = make_float4(inf, 0.f, -inf, 0.f);               // nothing is between
      if (rows && b >= 1 && b <= R) {
        const float l = __fdiv_rn((float)b - o, s) - d, h = __fdiv_rn((float)(b + 1) - o, s) + d;
        if (l >= u0 && h <= u1) {
          const float l0 = at(2 * ax, l), l1 = at(2 * ax, h), r0 = at(2 * ax + 1, l), r1 = at(2 * ax + 1, h);
          const float ml = __fdiv_rn(l1 - l0, h - l), mr = __fdiv_rn(r1 - r0, h - l);
          const float E = 3.814697265625e-06f;                   // 2^-18 = 64 u
          const float al = __fmaf_rn(-ml, l, l0) + E * __fmaf_rn(fabsf(ml), um, vm);
          const float ar = __fmaf_rn(-mr, l, r0) - E * __fmaf_rn(fabsf(mr), um, vm);
          if (fabsf(al) < inf && fabsf(ar) < inf && fabsf(ml) < 1.0e30f && fabsf(mr) < 1.0e30f)
            c = make_float4(al, ml, ar, mr);
        }
      }
      tab[ax * (R + 2) + b] = c;
      if (b == 0) { hdr->s[ax] = rows ? s : 0.f; hdr->o[ax] = rows ? o : 0.f; }
    }
    __threadfence();
  }
  cl_sync<CL>();
  return true;
}

// The header as another CTA of this kernel wrote it.
__device__ __forceinline__ SieveHdr fresh_hdr(const SieveHdr* h) {
  const float4 v = __ldcg(reinterpret_cast<const float4*>(h));
  return SieveHdr{{v.x, v.y}, {v.z, v.w}, 0u, 0u};
}

// Tables of each set from a sample spread over it in runs of 32 points, at most
// n / 8 of them.  What bounds it is a chain of dependent steps: of 26 us on 20M
// float64 points, 4 are the sample's loads, 3 its extremes, 7 the bands' minima,
// 1 the merge, 6 the peeling, 3 the chords and 2 the check at the end.  16 CTAs
// with 8 points per thread (8 with 16: 46 us); 131,072 points leave 23,600 of a
// 20M disk and 5,100 of a square; a sixteenth of the set instead of an eighth
// changed nothing below 2M points.
// A set of which the check finds too much left is refused (found out by k_refine
// instead, a circle took 23 to 31 us more); a fifth left (the degenerate kind) is
// listed up to kSetMax points, up to half of that in a batch, whose lists are one
// CTA's work each where it has many (96 degenerate sets of 60,000: 429 us refused,
// 787 listed).  A batch with a set per SM at most is sieved whole or not at all
// (Job::sv_all), so that it does not wait for lists and pipeline in turn (8
// degenerate sets of 38,000, half of them refused: 314 us, 209 so).
template <int DT, int R, int CL, int T, int NI>
__global__ void __launch_bounds__(T, kTabThreads / T) k_table(Job j, Ws w) {
  griddep_enter();
  extern __shared__ __align__(16) unsigned char smem[];
  TabSmem<R, T>& m = *reinterpret_cast<TabSmem<R, T>*>(smem);
  constexpr int W = T / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x % CL;
  const int set = blockIdx.x / CL;
  // a single set's control words: nothing of the call has touched them yet (a
  // memset in front of the kernel: 1 to 2 us more a call)
  if (CL > 1 && rank == 0) {
    constexpr uint32_t NW = sizeof(SetCtl) / 4;
    static_assert(sizeof(SetCtl) % 4 == 0, "whole words");
    for (uint32_t i = tid; i < NW + CT_COUNT; i += T) (i < NW ? reinterpret_cast<uint32_t*>(w.ctl) + i : w.ctr + (i - NW))[0] = 0u;
    for (uint32_t i = tid; i < (uint32_t)j.nchunkP; i += T) w.ptot[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  const SieveSet sd = j.sv_sets ? j.sv_sets[set] : j.sieve;
  SieveHdr* hdr = w.sv_hdr + set;
  float4* tab = w.sv_tab + (size_t)set * 2 * (R + 2);
  if (sd.nunit == 0) {                                 // uniform over the cluster
    if (rank == 0 && tid == 0) hdr->mode = 0;
    return;
  }
  // at most n / 8 points in runs of 32
  const int64_t groups = min((int64_t)CL * W * NI, max(sd.n / 256, (int64_t)1));
  const int64_t step = sd.n / groups;
  float X[NI], Y[NI];
  uint32_t valid = 0;
#pragma unroll
  for (int k = 0; k < NI; k++) {
    const int64_t g = ((int64_t)k * CL + rank) * W + warp;
    X[k] = Y[k] = 0.f;
    if (g < groups) valid |= (uint32_t)sieve_view<DT>(j, sd.off + g * step + lane, X[k], Y[k]) << k;
  }
  // the sample is here: k_sieve's CTAs may start and prefetch
  griddep_release();
  const bool ok = build_table<R, CL, T, NI>(m, X, Y, valid, rank, tab, hdr);
  // what is left of the sample (of 16384 points of it, 1024 of a batch's set)
  // tells whether the sieve pays
  constexpr int NC = CL > 1 ? 1 : kTabThreads / T;
  uint32_t outn = 0;
  if (ok) {
    const SieveHdr h = fresh_hdr(hdr);
#pragma unroll
    for (int k = 0; k < NC; k++) outn += ((valid >> k) & 1u) && !sieve_inside<R, true>(tab, h, X[k], Y[k]);
    outn = __reduce_add_sync(0xFFFFFFFFu, outn);
    if (lane == 0 && outn) atomicAdd(cl_map<CL>(&m.cnt, 0), outn);
    cl_sync<CL>();
  }
  if (rank == 0 && tid == 0) {
    const int64_t left = ok ? (int64_t)m.cnt * sd.n / (min(groups, (int64_t)CL * W * NC) * 32) : sd.n;
    hdr->mode = ok && left <= sd.cap ? 1u : 0u;
    if (hdr->mode == 0 && j.sv_all) w.ctr[CT_SIEVE_NONE] = 1u;
  }
}

constexpr int kSvThreads = kSvWarps * 32;
template <int DT>
constexpr int sv_items() { return DT == DT_F64 ? 4 : 8; }

// One warp per unit of consecutive points, two batches of loads in registers.
// float64 is bound by memory: 20M points in 55 us (5.8 TB/s), 46 behind k_table,
// which lets it prefetch 64 MB into L2 meanwhile (96 and 128 MB: the same).
// The 8-byte formats are bound by latency and the scattered reads of the table
// (11 shared wavefronts per 32 points): 20M float32 points in 44 us.  Slower: a
// four-stage cp.async ring per warp at 24 warps per SM (59 / 51 us), a box test
// before the table (149 against 143 us a call on the 20M square).
template <int DT, int R>
__global__ void __launch_bounds__(kSvThreads, 4) k_sieve(Job j, Ws w) {
  constexpr int U = sv_items<DT>();
  using V = RawPt<DT>;
  __shared__ float4 tab[2 * (R + 2)];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int set = j.sv_sets ? j.sv_cta[blockIdx.x] : 0;
  const SieveSet sd = j.sv_sets ? j.sv_sets[set] : j.sieve;
  const int64_t unit = (int64_t)(blockIdx.x - sd.cta0) * kSvWarps + warp;   // of the set
  const int64_t a0 = unit * sd.len;
  // before the table is there: the head of every unit into L2 (input only)
  if (a0 < sd.n) {
    const int64_t pre = min((int64_t)sd.pre, sd.n - a0);
    constexpr int B = DT == DT_F64 ? 16 : DT == DT_I32 ? 8 : 4;
    const char* p = reinterpret_cast<const char*>(j.pts) + (sd.off + a0) * B;
    for (int64_t q = lane * 128; q < pre * B; q += 32 * 128) asm volatile("prefetch.global.L2 [%0];" :: "l"(p + q));
    if constexpr (DT == DT_F32) {
      const char* y = reinterpret_cast<const char*>(j.ys + sd.off + a0);
      for (int64_t q = lane * 128; q < pre * B; q += 32 * 128) asm volatile("prefetch.global.L2 [%0];" :: "l"(y + q));
    }
  }
  griddep_enter();
  const SieveHdr hdr = w.sv_hdr[set];
  if (hdr.mode == 0 || (j.sv_all && w.ctr[CT_SIEVE_NONE] != 0)) return;
  for (int i = tid; i < 2 * (R + 2); i += kSvThreads) tab[i] = w.sv_tab[(size_t)set * 2 * (R + 2) + i];
  __syncthreads();
  if (a0 >= sd.n) return;
  const uint32_t cnt = (uint32_t)min((int64_t)sd.len, sd.n - a0);
  const uint32_t base = (uint32_t)a0;                   // set-local indices fit 32 bits
  uint32_t* out = w.valA + sd.off + a0;
  const V* src = reinterpret_cast<const V*>(j.pts) + sd.off + a0;
  const float* sx = reinterpret_cast<const float*>(j.pts) + sd.off + a0;
  const float* sy = j.ys + (DT == DT_F32 ? sd.off + a0 : 0);
  uint32_t nout = 0;
  V buf[2][U];
  auto load = [&](V (&b)[U], uint32_t i0) {
#pragma unroll
    for (int u = 0; u < U; u++) {
      const uint32_t i = i0 + u * 32 + lane;
      if (i < cnt) {
        if constexpr (DT == DT_F32) { b[u].x = __float_as_uint(__ldcs(sx + i)); b[u].y = __float_as_uint(__ldcs(sy + i)); }
        else b[u] = __ldcs(src + i);
      }
    }
  };
  auto test = [&](const V (&b)[U], uint32_t i0) {
    uint32_t left = 0;
#pragma unroll
    for (int u = 0; u < U; u++) {
      float X, Y;
      bool odd = false;
      if constexpr (DT == DT_F64) {
        // the views in f64_trunc_f32's bits; zeros, tiny, huge and NaN words
        // (unsigned wrap or a large exponent) are looked at again below
        const uint32_t tx = (b[u].y & 0x7FFFFFFFu) - 0x38000000u, ty = (b[u].w & 0x7FFFFFFFu) - 0x38000000u;
        odd = max(tx, ty) >= ((1023u + 60u) << 20) - 0x38000000u;
        X = __uint_as_float(__funnelshift_l(b[u].x, tx, 3) | (b[u].y & 0x80000000u));
        Y = __uint_as_float(__funnelshift_l(b[u].z, ty, 3) | (b[u].w & 0x80000000u));
      } else if constexpr (DT == DT_F32) {
        X = __uint_as_float(b[u].x);
        Y = __uint_as_float(b[u].y);
      } else {
        X = __int2float_rn((int)b[u].x);
        Y = __int2float_rn((int)b[u].y);
      }
      const bool in = sieve_between<R, false>(tab, hdr.s[0], hdr.o[0], Y, X);
      left |= (uint32_t)(!in | odd) << u;
    }
    if (__any_sync(0xFFFFFFFFu, left != 0)) {
#pragma unroll 1
      for (int u = 0; u < U; u++) {
        const uint32_t i = i0 + u * 32 + lane;
        bool l = ((left >> u) & 1u) && i < cnt;
        if (!__any_sync(0xFFFFFFFFu, l)) continue;
        if (l) {                                       // read again (unrolled on `b`: spills)
          float X, Y;
          l = !sieve_view<DT>(j, sd.off + a0 + i, X, Y) || !sieve_inside<R, false>(tab, hdr, X, Y);
        }
        const uint32_t bal = __ballot_sync(0xFFFFFFFFu, l);
        if (l) out[nout + __popc(bal & ((1u << lane) - 1u))] = base + i;
        nout += __popc(bal);
      }
    }
  };
  load(buf[0], 0);
  for (uint32_t i0 = 0; i0 < cnt; i0 += 2 * U * 32) {
    load(buf[1], i0 + U * 32);
    test(buf[0], i0);
    load(buf[0], i0 + 2 * U * 32);
    if (i0 + U * 32 < cnt) test(buf[1], i0 + U * 32);
  }
  if (lane == 0) w.sv_cnt[(size_t)blockIdx.x * kSvWarps + warp] = nout;
}

// Listed points of the set gathered in index order; outside the polygon of
// the listed points themselves where there are more than kPlain (20M disk:
// 23,600 to 2,300 in 30 us, the steps of k_table again; k_set on the longer list
// takes more than it saves -- with kPlain at 6144 the 20M square, 5,100 listed,
// went from 143 to 179 us).  Where the sample's polygon left more than a kLeast-th
// of the set, the listed points lie on the hull's own edge and their polygon drops
// few of them (degenerate set of 48,007, 9,600 listed: 124 us a call with the
// polygon, 104 without).
template <int DT, int R, int CL>
__global__ void __launch_bounds__(kTabThreads, 1) k_refine(Job j, Ws w) {
  griddep_enter();
  extern __shared__ __align__(16) unsigned char smem[];
  using M = TabSmem<R, kTabThreads>;
  M& m = *reinterpret_cast<M*>(smem);
  using P = typename PointT<DT>::T;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = blockIdx.x % CL;
  const SieveSet sd = j.sieve;
  SieveHdr* hdr = w.sv_hdr;
  float4* tab = w.sv_tab;
  if (hdr->mode == 0) return;                          // uniform over the cluster
  P* lp = reinterpret_cast<P*>(w.cpts);                // the list k_set reads
  uint32_t* li = w.cidx;
  // prefix over the units' counts, by every CTA
  const uint32_t nu = (uint32_t)sd.nunit;
  constexpr uint32_t PU = kSvMaxUnits / kTabThreads;
  uint32_t c[PU], sum = 0;
#pragma unroll
  for (uint32_t q = 0; q < PU; q++) {
    const uint32_t u = tid * PU + q;
    c[q] = u < nu ? w.sv_cnt[u] : 0u;
    sum += c[q];
  }
  uint32_t total = 0;
  {
    const uint32_t x = warp_incl_sum(sum);
    if (lane == 31) m.pre[warp] = x;
    __syncthreads();
    uint32_t pre = x - sum;
#pragma unroll
    for (int q = 0; q < M::W; q++) { const uint32_t v = m.pre[q]; pre += q < warp ? v : 0u; total += v; }
#pragma unroll
    for (uint32_t q = 0; q < PU; q++) { m.upre[tid * PU + q] = pre; pre += c[q]; }
    __syncthreads();
  }
  constexpr uint32_t kMost = CL * kTabThreads * kTabItems;
  if (total > kMost) return;                           // uniform: the pipeline takes the set
  // listed index number p
  auto listed = [&](uint32_t p) {
    uint32_t l = 0, h = kSvMaxUnits - 1;               // the last unit that starts at or before p
    while (l < h) {
      const uint32_t q = (l + h + 1) >> 1;
      if (m.upre[q] <= p) l = q; else h = q - 1;
    }
    return w.valA[sd.off + (int64_t)l * sd.len + (p - m.upre[l])];
  };
  if (total <= kPlain || (total <= (uint32_t)kSetMax && total > sd.n / kLeast)) {
    for (uint32_t i = rank * kTabThreads + tid; i < total; i += CL * kTabThreads) {
      const uint32_t g = listed(i);
      lp[i] = input_point<P>(j, sd.off + g);
      li[i] = g;
    }
    if (rank == 0 && tid == 0) { hdr->n = total; w.ctr[CT_SIEVED] = 1u; }
    return;
  }
  // items in index order: CTA, warp, k, lane
  const uint32_t cper = ((total + CL - 1) / CL + 31) / 32 * 32;           // per CTA
  const uint32_t wper = ((cper + M::W - 1) / M::W + 31) / 32 * 32;   // per warp: 32 kTabItems at most
  const uint32_t w0 = rank * cper + warp * wper;
  const uint32_t w1 = min(min(total, (uint32_t)(rank + 1) * cper), w0 + wper);
  uint32_t g[kTabItems];
  float X[kTabItems], Y[kTabItems];
  uint32_t valid = 0, have = 0;
#pragma unroll
  for (int k = 0; k < kTabItems; k++) {
    const uint32_t i = w0 + k * 32 + lane;
    g[k] = i < w1 ? listed(i) : 0u;
    have |= (uint32_t)(i < w1) << k;
  }
#pragma unroll
  for (int k = 0; k < kTabItems; k++) {
    X[k] = Y[k] = 0.f;
    if ((have >> k) & 1u) valid |= (uint32_t)sieve_view<DT>(j, sd.off + g[k], X[k], Y[k]) << k;
  }
  const bool ok = build_table<R, CL, kTabThreads, kTabItems>(m, X, Y, valid, rank, tab, hdr);
  uint32_t keep = have;
  if (ok) {
    const SieveHdr h = fresh_hdr(hdr);
#pragma unroll
    for (int k = 0; k < kTabItems; k++)
      if (((valid >> k) & 1u) && sieve_inside<R, true>(tab, h, X[k], Y[k])) keep &= ~(1u << k);
  }
  // stable compaction: counts per warp, per CTA, over the cluster
  uint32_t wc = 0;
#pragma unroll
  for (int k = 0; k < kTabItems; k++) wc += __popc(__ballot_sync(0xFFFFFFFFu, (keep >> k) & 1u));
  if (lane == 0) m.pre[warp] = wc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t v = __reduce_add_sync(0xFFFFFFFFu, m.pre[lane]);
    if (lane == 0) m.cnt = v;                          // this CTA's count
  }
  cl_sync<CL>();
  uint32_t pos = 0, m2 = 0;
#pragma unroll
  for (int q = 0; q < CL; q++) { const uint32_t v = *cl_map<CL>(&m.cnt, q); pos += q < rank ? v : 0u; m2 += v; }
  for (int q = 0; q < warp; q++) pos += m.pre[q];
  if (m2 <= (uint32_t)kSetMax) {                       // uniform over the cluster
#pragma unroll
    for (int k = 0; k < kTabItems; k++) {
      const bool kp = (keep >> k) & 1u;
      const uint32_t bal = __ballot_sync(0xFFFFFFFFu, kp);
      if (kp) {
        const uint32_t p = pos + __popc(bal & ((1u << lane) - 1u));
        lp[p] = input_point<P>(j, sd.off + g[k]);
        li[p] = g[k];
      }
      pos += __popc(bal);
    }
    if (rank == 0 && tid == 0) { hdr->n = m2; w.ctr[CT_SIEVED] = 1u; }
  }
  cl_sync<CL>();                                       // nobody leaves while its count is read
}

constexpr int kSvCluster = 16;                     // CTAs per cluster (more than 8: opt-in)
constexpr int64_t kSvPrefetch = int64_t(64) << 20;  // bytes k_sieve prefetches while k_table runs

// Clusters of kernel fn (attributes set) that fit the device at once.
int clusters_resident(const void* fn, size_t smem) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = kSvCluster;
  cfg.blockDim = kTabThreads;
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kSvCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
  return n;
}

// Sets the single-set kernels' attributes; whether their clusters can run here.
template <int DT>
bool sieve_fits() {
  constexpr size_t sm = sizeof(TabSmem<kSvRows, kTabThreads>), smr = sizeof(TabSmem<kSvRefineRows, kTabThreads>);
  static const bool ok = [] {
    auto* t = k_table<DT, kSvRows, kSvCluster, kTabThreads, kTabItems>;
    auto* r = k_refine<DT, kSvRefineRows, kSvCluster>;
    cudaFuncSetAttribute(t, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    cudaFuncSetAttribute(t, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaFuncSetAttribute(r, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smr);
    cudaFuncSetAttribute(r, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return clusters_resident((const void*)t, sm) > 0 && clusters_resident((const void*)r, smr) > 0;
  }();
  return ok;
}

template <int DT>
int launch_table_t(const Job& j, const Ws& w, int sms, cudaStream_t st) {
  constexpr int T = kTabThreads, TB = kTabBatchThreads, CL = kSvCluster, R = kSvRows, RB = kSvBatchRows;
  constexpr size_t sm = sizeof(TabSmem<R, T>), smb = sizeof(TabSmem<RB, TB>), smf = sizeof(TabSmem<RB, T>);
  if (j.sv_sets) {
    static bool once = [] {
      cudaFuncSetAttribute(k_table<DT, RB, 1, TB, kTabBatchItems>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smb);
      cudaFuncSetAttribute(k_table<DT, RB, 1, T, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smf);
      return true;
    }();
    (void)once;
    if (j.nsets <= sms / 2) launch_pdl(k_table<DT, RB, 1, T, 4>, j.nsets, T, smf, st, j, w);
    else launch_pdl(k_table<DT, RB, 1, TB, kTabBatchItems>, j.nsets, TB, smb, st, j, w);
    return 1;
  }
  launch_pdl_cluster(k_table<DT, R, CL, T, kTabItems>, CL, T, CL, sm, st, j, w);
  return 1;
}

template <int DT>
int launch_sieve_t(const Job& j, const Ws& w, cudaStream_t st) {
  static_assert(kSvRows == kSvBatchRows, "one k_sieve for both");
  const int grid = j.sv_sets ? j.sv_nctas : (j.sieve.nunit + kSvWarps - 1) / kSvWarps;
  launch_pdl(k_sieve<DT, kSvRows>, grid, kSvThreads, 0, st, j, w);
  return 1;
}

template <int DT>
int launch_refine_t(const Job& j, const Ws& w, cudaStream_t st) {
  constexpr int CL = kSvCluster, R = kSvRefineRows;
  constexpr size_t sm = sizeof(TabSmem<R, kTabThreads>);
  launch_pdl_cluster(k_refine<DT, R, CL>, CL, kTabThreads, CL, sm, st, j, w);
  return 1;
}

}  // namespace

SieveSet sieve_set(int64_t off, int64_t n, int dtype, int sms) {
  const int64_t step = 32 * (dtype == DT_F64 ? sv_items<DT_F64>() : sv_items<DT_I32>());
  const int64_t most = std::min<int64_t>((int64_t)sms * 4 * kSvWarps, kSvMaxUnits);
  SieveSet s{};
  if (!(dtype == DT_F64 ? sieve_fits<DT_F64>() : dtype == DT_F32 ? sieve_fits<DT_F32>() : sieve_fits<DT_I32>())) return s;
  s.off = off;
  s.n = n;
  s.len = ((n + most - 1) / most + step - 1) / step * step;
  s.nunit = (int32_t)((n + s.len - 1) / s.len);
  s.pre = (int32_t)std::min<int64_t>(s.len, kSvPrefetch / ((dtype == DT_F64 ? 16 : 8) * (int64_t)s.nunit));
  static_assert(kSvCluster * kTabThreads * kTabItems == kSvMost, "a thread holds kTabItems listed points");
  s.cap = std::min(kSvMost, std::max<int64_t>(n / kLeast, kSetMax));
  return s;
}

SieveSet sieve_batch_set(int64_t off, int64_t n, int32_t cta0, int32_t most) {
  SieveSet s{};
  s.off = off;
  s.n = n;
  s.len = kSvBatchLen;
  const int64_t units = (n + kSvBatchLen - 1) / kSvBatchLen;
  s.nunit = units <= most ? (int32_t)units : 0;
  s.cap = std::min<int64_t>(kSetMax / 4 * 3, std::max<int64_t>(n / kLeast, kSetMax / 2));
  s.cta0 = cta0;
  return s;
}

int launch_table(const Job& j, const Ws& w, int sms, cudaStream_t st) {
  return j.dtype == DT_F64 ? launch_table_t<DT_F64>(j, w, sms, st)
         : j.dtype == DT_F32 ? launch_table_t<DT_F32>(j, w, sms, st) : launch_table_t<DT_I32>(j, w, sms, st);
}

int launch_sieve(const Job& j, const Ws& w, cudaStream_t st) {
  return j.dtype == DT_F64 ? launch_sieve_t<DT_F64>(j, w, st)
         : j.dtype == DT_F32 ? launch_sieve_t<DT_F32>(j, w, st) : launch_sieve_t<DT_I32>(j, w, st);
}

int launch_refine(const Job& j, const Ws& w, cudaStream_t st) {
  if (j.sv_sets) return 0;
  return j.dtype == DT_F64 ? launch_refine_t<DT_F64>(j, w, st)
         : j.dtype == DT_F32 ? launch_refine_t<DT_F32>(j, w, st) : launch_refine_t<DT_I32>(j, w, st);
}

}  // namespace cch
