// hull_block.cuh -- steps 4-7 of Sec. 2.1 for one set whose region points fit
// one CTA: dominance filter, Table 1 sort, Fig. 2 SPA, the simple polygon and
// its strictly convex hull, from a list of candidates in shared memory to the
// set's output indices.
//
// A candidate is a 14-bit number c (kBlkMax = 2^14 at most) and a region
// r = 0..3, packed r << 14 | c; a source object turns c into the exact point
// and the output index.  Candidate order must be index order (ties in the sort
// go to the smaller c).  Points are read through the source (L1 / L2 hits:
// a set is at most 256 KB), so shared memory holds 16-bit lists only and
// several CTAs share an SM; what bounds the block is the latency of its dozen
// dependent steps, which the other CTAs of the SM fill.
#pragma once
#include "chain.cuh"
#include "round1.cuh"

namespace cch {

constexpr int kBlkMax = 16384;          // candidate numbers are below it (14 bits); a block takes fewer than
                                        // CAP <= kBlkMax points, so no entry is 0xFFFF, the sort's padding
// Ranking a bucket compares its members pair by pair, sum(occ^2) comparisons in
// all; above kBlkPairs per kept candidate (many equal keys) the candidates behind
// their bucket's best one go first, and a bitonic sort of log2(m)^2 / 2 passes
// takes the rest.
constexpr uint32_t kBlkPairs = 128;
constexpr uint32_t kBlkCrowd = 1024;    // so many candidates are sorted without that (3M int32 square points, some
                                        // hundred in one bucket: 70 us a call, 73 with it)
constexpr uint16_t kPin = 0x8000u;      // polygon entry that is one of E1..E4

// Set-wide values of a block, in shared memory.
template <int DT>
struct BlkSet {
  using P = typename PT<DT>::T;
  P e[4];                    // E1..E4
  double ex[4], ey[4];       // the same, as the exact region tests take them
  uint32_t eidx[4];          // candidate numbers of E1..E4
  uint64_t v0[4];            // SPA value of E_r
  float lo[4], sc[4];        // bucket map of region r
  uint32_t down;             // exponent that blk_view takes off (word's bits)
  float fA[4], fB[4], fC[4], fE[4];   // FP32 filter of edge r (round1.cuh)
  uint32_t flags;
  int status;
};

template <int DT, int CAP, int T, int NB>
struct BlkSmem {
  static_assert(CAP <= kBlkMax && 4 * NB % T == 0 && T % 128 == 0, "whole buckets per thread, whole warps per region");
  static_assert((CAP + 1 + 2 * T) * 2 <= 2 * 4 * NB * 4, "links, heads and tails of the bridge walks fit tab and cnt");
  static_assert(CAP / T <= 32, "a thread's share of the candidates fits a 32-bit mask");
  uint16_t a[CAP + 8];       // candidate list, bucket members, polygon
  uint16_t b[CAP + 8];       // kept candidates, sorted order, polygon (ping-pong)
  uint32_t tab[4 * NB];      // per region and bucket: smallest leading SPA word, then its exclusive prefix minimum
  uint32_t cnt[4 * NB + 8];  // kept candidates per bucket, then bucket starts and ends
  uint32_t dead[CAP / 32 + 1];
  BlkSet<DT> s;
  uint64_t w64[T / 32];
  int wreg[T / 32];
  uint32_t w32[2][T / 32];
  uint32_t n[4];             // list lengths
  unsigned long long s2;     // SPA survivors per region, 16 bits each
  uint32_t hn, hb;           // the hull's vertices and the list that holds them (0: a, 1: b)
  uint32_t close;            // candidate number of the point that closes the polygon
};

// Sort key and SPA value of a point of region r (0..3), Table 1 / Fig. 2.
template <int DT>
__device__ __forceinline__ uint64_t blk_key(const typename PT<DT>::T& p, int r) {
  if constexpr (DT == DT_F64) {
    const uint64_t k = key_f64((uint64_t)__double_as_longlong((r & 1) ? p.y : p.x));
    return r >= 2 ? ~k : k;
  } else {
    const uint64_t k = key_i32((r & 1) ? p.y : p.x);
    return r >= 2 ? k ^ 0xFFFFFFFFull : k;
  }
}
template <int DT>
__device__ __forceinline__ uint64_t blk_spa(const typename PT<DT>::T& p, int r) {
  const bool neg = r == 1 || r == 2;
  if constexpr (DT == DT_F64) {
    const uint64_t k = key_f64((uint64_t)__double_as_longlong((r & 1) ? p.x : p.y));
    return neg ? ~k : k;
  } else {
    const uint64_t k = key_i32((r & 1) ? p.x : p.y);
    return neg ? k ^ 0xFFFFFFFFull : k;
  }
}
// Leading 32 bits of an SPA value: strictly larger means strictly worse.
template <int DT>
__device__ __forceinline__ uint32_t blk_word(uint64_t v) {
  return DT == DT_F64 ? (uint32_t)(v >> 32) : (uint32_t)v;
}

// FP32 view of a sort coordinate for the bucket map.  float64 coordinates of a
// set beyond 2^60 get 2^-down first, which brings the largest to [1, 2) and
// what would leave the normal range to 0; non-decreasing in the coordinate.
template <int DT>
__device__ __forceinline__ float blk_view(const BlkSet<DT>& s, const typename PT<DT>::T& p, int r) {
  if constexpr (DT == DT_F64) {
    uint64_t b = (uint64_t)__double_as_longlong((r & 1) ? p.y : p.x);
    if (!(s.flags & SF_SMALL)) {
      const uint32_t h = (uint32_t)(b >> 32);
      b = (h & 0x7FF00000u) > s.down ? b - ((uint64_t)s.down << 32) : b & 0x8000000000000000ull;
    }
    return f64_trunc_f32(b);
  } else {
    return __int2float_rn((r & 1) ? p.y : p.x);
  }
}

// Bucket of a region-r point, non-decreasing in its sort key.
template <int DT, int NB>
__device__ __forceinline__ int blk_bucket(const BlkSet<DT>& s, const typename PT<DT>::T& p, int r) {
  const float u = blk_view<DT>(s, p, r);
  const float t = __fmul_rn(__fsub_rn(r >= 2 ? -u : u, s.lo[r]), s.sc[r]);
  return min(max(__float2int_rd(t), 0), NB - 1);
}

// Bucket map and SPA seed of region r (e, flags and down are set).
template <int DT, int NB>
__device__ __forceinline__ void blk_map(BlkSet<DT>& s, int r) {
  const typename PT<DT>::T p = s.e[r], q = s.e[(r + 1) & 3];
  s.v0[r] = blk_spa<DT>(p, r);
  const float sg = r >= 2 ? -1.f : 1.f, lo = sg * blk_view<DT>(s, p, r), d = __fsub_rn(sg * blk_view<DT>(s, q, r), lo);
  const float sc = d > 0.f ? __fdiv_rn((float)NB, d) : 0.f;
  s.lo[r] = lo;
  s.sc[r] = sc <= 1.0e38f ? sc : 1.0e38f;
}

// Barrier of the T threads that run a step: the CTA, or its first warp alone.
template <int T>
__device__ __forceinline__ void blk_sync() {
  if constexpr (T == 32) __syncwarp();
  else __syncthreads();
}

// Exclusive prefix sum of one value per thread; `tot` receives the sum.  One
// barrier; `sh` alternates between calls (the caller passes 0, 1, 0, ...), so
// the next call's writes cannot meet this call's reads.
template <int T>
__device__ __forceinline__ uint32_t blk_excl_sum(uint32_t v, uint32_t* sh, uint32_t& tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if constexpr (T == 32) {
    __syncwarp();                        // orders the caller's shared accesses like the barrier below
    tot = __shfl_sync(0xFFFFFFFFu, x, 31);
    return x - v;
  }
  if (lane == 31) sh[warp] = x;
  __syncthreads();
  uint32_t pre = x - v, t = 0;
#pragma unroll
  for (int q = 0; q < T / 32; q++) {
    const uint32_t c = sh[q];
    if (q < warp) pre += c;
    t += c;
  }
  tot = t;
  return pre;
}

// Append the entries with a set bit in `take` (bit u: v[u]) of every lane to a
// list, in any order, with one atomic per warp; every lane calls it.
template <int U>
__device__ __forceinline__ void blk_append(uint16_t* list, uint32_t* n, uint32_t take, const uint32_t (&v)[U]) {
  const int lane = threadIdx.x & 31;
  const uint32_t c = __popc(take);
  uint32_t x = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  uint32_t base = 0;
  if (lane == 31 && x) base = atomicAdd(n, x);
  base = __shfl_sync(0xFFFFFFFFu, base, 31) + x - c;
#pragma unroll
  for (int u = 0; u < U; u++)
    if ((take >> u) & 1u) list[base++] = (uint16_t)v[u];
}

// Orientation of three polygon points: the FP32 filter on their views, the
// split points only where it leaves the sign open (float64; int32 exactly).
template <int DT>
__device__ __forceinline__ int blk_orient(const typename PT<DT>::T& a, const typename PT<DT>::T& b,
                                          const typename PT<DT>::T& c, bool flag) {
  if constexpr (DT == DT_F64) {
    if (flag) {
      float2 A, B, C;
      f32_view<DT>(a, A.x, A.y);
      f32_view<DT>(b, B.x, B.y);
      f32_view<DT>(c, C.x, C.y);
      int o = orient_f32_filter(A, B, C);
      if (o) return o;
      o = orient_split_filter(f64_split4(a), f64_split4(b), f64_split4(c));
      if (o) return o;
    }
    return orient_f64(a.x, a.y, b.x, b.y, c.x, c.y, flag);
  } else {
    return orient_i32(a.x, a.y, b.x, b.y, c.x, c.y, flag);
  }
}

// Polygon points by position, for the bridge walks.
template <int DT, class Src>
struct BlkAcc {
  const Src& src;
  const uint16_t* cur;
  uint16_t *pv, *nx;
  uint32_t* dead;
  bool flag;
  __device__ __forceinline__ int prv(int i) const { return pv[i]; }
  __device__ __forceinline__ int nxt(int i) const { return nx[i]; }
  __device__ __forceinline__ void kill(int i) { atomicOr(dead + (i >> 5), 1u << (i & 31)); }
  __device__ __forceinline__ void link(int x, int y) { nx[x] = (uint16_t)y; pv[y] = (uint16_t)x; }
  __device__ __forceinline__ int orient(int i, int j, int k) const {
    return blk_orient<DT>(src.pt(cur[i] & ~kPin), src.pt(cur[j] & ~kPin), src.pt(cur[k] & ~kPin), flag);
  }
};

// Strictly convex hull of the closed polygon cur[0..L) (first point repeated
// last; every other entry different from its predecessor), kept entries in
// order at the start of the returned buffer, their number in L.  Peeling: an
// entry without a strict left turn between its current neighbours lies on or
// inside a segment of two polygon points, so it is no strict vertex, and all
// such entries go at once, round after round; E1..E4 stay (they are vertices;
// between coincident or collinear points no turn would show it).  A polygon
// that has not settled in kPeelRounds rounds (a long convex run undone from
// one end) is finished by one strict left-turn stack per thread over its
// share of the entries and pairwise bridge walks; `lnk` holds 2 links per
// entry.
template <int DT, int T, class Src>
__device__ uint16_t* blk_hull(const Src& src, uint16_t* cur, uint16_t* nxt, uint16_t* lnk, uint32_t* dead,
                              uint32_t* sh0, uint32_t* sh1, bool flag, uint32_t& L) {
  using P = typename PT<DT>::T;
  const int tid = threadIdx.x;            // < T
  uint32_t n = L;
  bool conv = false;
  for (int round = 0; round < kPeelRounds && !conv; round++) {
    const uint32_t per = (n + T - 1) / T, t0 = tid * per, t1 = min(n, t0 + per);
    uint64_t keep = 0;
    if (t0 < t1) {
      P p[3];
      p[0] = src.pt(cur[t0 ? t0 - 1 : 0] & ~kPin);
      p[1] = src.pt(cur[t0] & ~kPin);
#pragma unroll 1
      for (uint32_t t = t0; t < t1; t++) {
        p[2] = src.pt(cur[min(t + 1, n - 1)] & ~kPin);
        const bool k = (cur[t] & kPin) || blk_orient<DT>(p[0], p[1], p[2], flag) > 0;
        keep |= (uint64_t)k << (t - t0);
        p[0] = p[1]; p[1] = p[2];
      }
    }
    uint32_t n2;
    uint32_t pre = blk_excl_sum<T>((uint32_t)__popcll((long long)keep), (round & 1) ? sh1 : sh0, n2);
    conv = n2 == n;                      // uniform
    if (!conv) {
      for (uint32_t t = t0; t < t1; t++)
        if ((keep >> (t - t0)) & 1u) nxt[pre++] = cur[t];
      n = n2;
      uint16_t* x = cur; cur = nxt; nxt = x;
      blk_sync<T>();
    }
  }
  if (!conv) {
    uint16_t* pv = lnk;
    uint16_t* nx = nxt;
    uint16_t* hd = lnk + n;              // chain head and tail per thread
    uint16_t* tl = hd + T;
    BlkAcc<DT, Src> acc{src, cur, pv, nx, dead, flag};
    for (uint32_t i = tid; i < (n + 31) / 32; i += T) dead[i] = 0;
    blk_sync<T>();
    const uint32_t per = (n + T - 1) / T, t0 = tid * per, t1 = min(n, t0 + per);
    // the stack lives in the links: its top is `top`, below it pv[top]
    int head = -1, top = -1;
    for (uint32_t t = t0; t < t1; t++) {
      while (top >= 0 && top != head && acc.orient(pv[top], top, (int)t) <= 0) { acc.kill(top); top = pv[top]; }
      if (top >= 0) acc.link(top, (int)t); else head = (int)t;
      top = (int)t;
    }
    hd[tid] = (uint16_t)(head < 0 ? 0xFFFF : head);
    tl[tid] = (uint16_t)(top < 0 ? 0xFFFF : top);
    for (int step = 1; step < T; step <<= 1) {
      blk_sync<T>();
      if ((tid & (2 * step - 1)) == 0 && tid + step < T) {
        int hl = hd[tid] == 0xFFFF ? -1 : hd[tid], ta = tl[tid];
        const int hr = hd[tid + step] == 0xFFFF ? -1 : hd[tid + step];
        merge_chains(acc, hl, ta, hr, (int)tl[tid + step]);
        if (hl >= 0) { hd[tid] = (uint16_t)hl; tl[tid] = (uint16_t)ta; }
      }
    }
    blk_sync<T>();
    // compact the kept entries (the links are dead: nxt is free)
    uint64_t keep = 0;
    for (uint32_t t = t0; t < t1; t++) keep |= (uint64_t)(!((dead[t >> 5] >> (t & 31)) & 1u)) << (t - t0);
    uint32_t n2;
    uint32_t pre = blk_excl_sum<T>((uint32_t)__popcll((long long)keep), sh0, n2);
    for (uint32_t t = t0; t < t1; t++)
      if ((keep >> (t - t0)) & 1u) nxt[pre++] = cur[t];
    n = n2;
    cur = nxt;
    blk_sync<T>();
  }
  L = n;
  return cur;
}

// From the sorted candidates m.b[0 .. m2) to the hull (m.hn, m.hb), by the
// first T threads of the CTA.
template <int DT, int T, class M, class Src>
__device__ void blk_tail(M& m, const Src& src, uint32_t m2) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const BlkSet<DT>& s = m.s;
  // SPA: exclusive prefix minimum of the SPA value within each region,
  // seeded with E_r; the scan carries (last region, its minimum)
  const uint32_t per = (m2 + T - 1) / T, i0 = min(m2, tid * per), i1 = min(m2, i0 + per);
  int reg = -1;
  uint64_t mn = ~0ull;
  for (uint32_t i = i0; i < i1; i++) {
    const uint32_t e = m.b[i];
    const int r = (int)(e >> 14);
    const uint64_t v = blk_spa<DT>(src.pt(e & 0x3FFFu), r);
    mn = r == reg ? min(mn, v) : v;
    reg = r;
  }
  int xr = reg;
  uint64_t xm = mn;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int yr = __shfl_up_sync(0xFFFFFFFFu, xr, o);
    const uint64_t ym = __shfl_up_sync(0xFFFFFFFFu, xm, o);
    if (lane >= o) {
      if (yr > xr) { xr = yr; xm = ym; }
      else if (yr == xr) xm = min(xm, ym);
    }
  }
  if (lane == 31) { m.w64[warp] = xm; m.wreg[warp] = xr; }
  blk_sync<T>();
  int pr = __shfl_up_sync(0xFFFFFFFFu, xr, 1);
  uint64_t pm = __shfl_up_sync(0xFFFFFFFFu, xm, 1);
  if (lane == 0) { pr = -1; pm = ~0ull; }
  for (int q = warp - 1; q >= 0; q--) {
    const int yr = m.wreg[q];
    if (yr > pr) { pr = yr; pm = m.w64[q]; }
    else if (yr == pr) pm = min(pm, m.w64[q]);
    else break;
  }
  uint32_t keep = 0;
  unsigned long long c4 = 0;                  // kept per region
  for (uint32_t i = i0; i < i1; i++) {
    const uint32_t e = m.b[i];
    const int r = (int)(e >> 14);
    const uint64_t v = blk_spa<DT>(src.pt(e & 0x3FFFu), r);
    if (r != pr) { pr = r; pm = s.v0[r]; }
    else pm = min(pm, s.v0[r]);
    if (v <= pm) { keep |= 1u << (i - i0); c4 += 1ull << (16 * r); }
    pm = min(pm, v);
  }
  {
    const uint32_t lo = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)c4), hi = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(c4 >> 32));
    if (lane == 0 && (lo | hi)) atomicAdd(&m.s2, ((unsigned long long)hi << 32) | lo);
  }
  uint32_t tot;
  uint32_t pre = blk_excl_sum<T>((uint32_t)__popc(keep), m.w32[0], tot);
  // the simple polygon: per region with E_r != E_{r+1}, E_r and the
  // survivors in order; closed by m.close (the first point again)
  const uint32_t flags = s.flags;
  uint32_t L = tot + 1;
#pragma unroll
  for (int r = 0; r < 4; r++) L += !(flags & (SF_DEGEN0 << r));
  if (L == 1) {                               // every point identical
    if (tid == 0) { m.a[0] = (uint16_t)s.eidx[0]; m.hn = 1; m.hb = 0; }
    return;
  }
  for (uint32_t i = i0; i < i1; i++) {
    if (!((keep >> (i - i0)) & 1u)) continue;
    const uint32_t e = m.b[i];
    uint32_t o = pre++;
#pragma unroll
    for (int r = 0; r < 4; r++) o += (uint32_t)r <= (e >> 14) && !(flags & (SF_DEGEN0 << r));
    m.a[o] = (uint16_t)(e & 0x3FFFu);
  }
  if (tid == 0) {
    const unsigned long long s2 = m.s2;       // complete: blk_excl_sum synchronised after the adds
    uint32_t o = 0;
#pragma unroll
    for (int r = 0; r < 4; r++) {
      if (!(flags & (SF_DEGEN0 << r))) {
        m.a[o++] = (uint16_t)(s.eidx[r] | kPin);
      }
      o += (uint32_t)(s2 >> (16 * r)) & 0xFFFFu;
    }
    m.a[o] = (uint16_t)(m.close | kPin);
  }
  blk_sync<T>();
  // identical neighbours: the first (smallest index) stays
  uint32_t L2;
  {
    const uint32_t pl = (L + T - 1) / T, t0 = min(L, tid * pl), t1 = min(L, t0 + pl);
    uint64_t kp = 0;
    for (uint32_t t = t0; t < t1; t++) {
      const uint32_t e = m.a[t];
      const bool k = (e & kPin) || !same_pt<DT>(src.pt(e), src.pt(m.a[t - 1] & ~kPin));
      kp |= (uint64_t)k << (t - t0);
    }
    uint32_t o = blk_excl_sum<T>((uint32_t)__popcll((long long)kp), m.w32[1], L2);
    for (uint32_t t = t0; t < t1; t++)
      if ((kp >> (t - t0)) & 1u) m.b[o++] = m.a[t];
  }
  blk_sync<T>();
  const bool flag = DT == DT_F64 ? (flags & SF_SMALL) != 0 : (flags & SF_WIDE) != 0;
  const uint16_t* h = blk_hull<DT, T>(src, m.b, m.a, reinterpret_cast<uint16_t*>(m.tab), m.dead, m.w32[0], m.w32[1], flag, L2);
  if (tid == 0) { m.hn = L2 - 1; m.hb = h == m.b; }
}

// Most sorted candidates that one warp takes to the end alone: it needs no
// CTA barriers (its steps have at most 8 entries per lane), and the CTA's
// other warps leave.
constexpr uint32_t kBlkWarpTail = 256;

// Steps 4-7 from the candidate list m.a[0 .. m.n[0]) to the hull (m.hn, m.hb;
// not synchronised).  On entry
// m.tab holds the smallest leading SPA word of the set's region-r points per
// bucket (any subset of them), m.cnt and m.n[1..], m.s2 are zero, and the CTA
// is synchronised.
template <int DT, int CAP, int T, int NB, class Src>
__device__ void blk_finish(BlkSmem<DT, CAP, T, NB>& m, const Src& src) {
  using P = typename PT<DT>::T;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int Q = 4 * NB / T;               // buckets per thread
  const BlkSet<DT>& s = m.s;
  // exclusive prefix minimum per region, seeded with E_r's word
  {
    const int r = tid / (T / 4);
    uint32_t loc = 0xFFFFFFFFu;
#pragma unroll
    for (int q = 0; q < Q; q++) loc = min(loc, m.tab[tid * Q + q]);
    uint32_t x = loc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x = min(x, y);
    }
    if (lane == 31) m.w32[0][warp] = x;
    __syncthreads();
    uint32_t run = __shfl_up_sync(0xFFFFFFFFu, x, 1);
    if (lane == 0) run = 0xFFFFFFFFu;
    for (int q = r * (T / 128); q < warp; q++) run = min(run, m.w32[0][q]);
    run = min(run, blk_word<DT>(s.v0[r]));
#pragma unroll
    for (int q = 0; q < Q; q++) {
      const uint32_t v = m.tab[tid * Q + q];
      m.tab[tid * Q + q] = run;
      run = min(run, v);
    }
  }
  __syncthreads();
  // a candidate that a point of a strictly lower bucket beats strictly is no
  // SPA survivor; the others are counted per bucket
  const uint32_t mc = m.n[0];
  for (uint32_t t0 = 0; t0 < mc; t0 += 4 * T) {
    uint32_t e[4], keep = 0;
    P p[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const uint32_t t = t0 + u * T + tid;
      e[u] = t < mc ? m.a[t] : 0u;
      if (t < mc) p[u] = src.pt(e[u] & 0x3FFFu);
    }
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (t0 + u * T + tid < mc) {
        const int r = (int)(e[u] >> 14);
        const int b = r * NB + blk_bucket<DT, NB>(s, p[u], r);
        if (blk_word<DT>(blk_spa<DT>(p[u], r)) <= m.tab[b]) {
          keep |= 1u << u;
          atomicAdd(&m.cnt[b], 1u);
        }
      }
    }
    blk_append(m.b, &m.n[1], keep, e);
  }
  __syncthreads();
  uint32_t m2 = m.n[1];
  if (m2 != 0) {                              // uniform
    // bucket starts
    {
      uint32_t loc[Q], sum = 0, pairs = 0;
#pragma unroll
      for (int q = 0; q < Q; q++) { loc[q] = m.cnt[tid * Q + q]; sum += loc[q]; pairs += loc[q] * loc[q]; }
      pairs = __reduce_add_sync(0xFFFFFFFFu, pairs);
      if (lane == 0 && pairs) atomicAdd(&m.n[2], pairs);
      uint32_t tot;
      uint32_t pre = blk_excl_sum<T>(sum, m.w32[1], tot);
#pragma unroll
      for (int q = 0; q < Q; q++) { m.cnt[tid * Q + q] = pre; pre += loc[q]; }
    }
    __syncthreads();
    if (m.n[2] <= kBlkPairs * m2) {           // sum(occ^2) <= 2^28: no overflow
      // counting sort by bucket, then the rank within the bucket by (key, c)
      for (uint32_t t = tid; t < m2; t += T) {
        const uint32_t e = m.b[t];
        const int r = (int)(e >> 14);
        const int b = r * NB + blk_bucket<DT, NB>(s, src.pt(e & 0x3FFFu), r);
        m.a[atomicAdd(&m.cnt[b], 1u)] = (uint16_t)e;   // the start becomes the bucket's end
      }
      __syncthreads();
      for (uint32_t t = tid; t < m2; t += T) {
        const uint32_t e = m.a[t];
        const int r = (int)(e >> 14);
        const P p = src.pt(e & 0x3FFFu);
        const int b = r * NB + blk_bucket<DT, NB>(s, p, r);
        const uint64_t k = blk_key<DT>(p, r);
        const uint32_t st = b ? m.cnt[b - 1] : 0u, en = m.cnt[b];
        uint32_t rank = 0;
        for (uint32_t x = st; x < en; x++) {
          const uint32_t f = m.a[x];
          const uint64_t kf = blk_key<DT>(src.pt(f & 0x3FFFu), r);
          rank += (kf < k) || (kf == k && f < e);
        }
        m.b[st + rank] = (uint16_t)e;
      }
    } else {
      // Crowded buckets (equal or nearly equal keys: a flat side, copies).  With
      // f the bucket's smallest by (SPA value, key, c), another candidate e
      // whose key is not below f's is no vertex: the line from f through e
      // (right of f or level, above it or level, in region 1's terms) meets the
      // segment E_r E_{r+1} behind e, which is outside it; a copy of f has a
      // larger index.  Then a bitonic sort of what is left by (region, key, c),
      // the pad entries 0xFFFF last.  (2M points on an 801 x 801 grid, 10,000
      // of them listed from its sides: 316 us a call by the sort alone, 155 so.)
      if (CAP > 2 * kBlkCrowd && m2 > kBlkCrowd) {
        for (uint32_t t = tid; t < 4 * NB; t += T) m.tab[t] = 0xFFFFFFFFu;
        __syncthreads();
        for (uint32_t t = tid; t < m2; t += T) {
          const uint32_t e = m.b[t];
          const int r = (int)(e >> 14);
          const P p = src.pt(e & 0x3FFFu);
          const uint64_t v = blk_spa<DT>(p, r), k = blk_key<DT>(p, r);
          uint32_t* best = &m.tab[r * NB + blk_bucket<DT, NB>(s, p, r)];
          uint32_t f = *(volatile uint32_t*)best;
          for (;;) {
            if (f != 0xFFFFFFFFu) {
              const P q = src.pt(f & 0x3FFFu);
              const uint64_t vf = blk_spa<DT>(q, r), kf = blk_key<DT>(q, r);
              if (vf < v || (vf == v && (kf < k || (kf == k && f < e)))) break;
            }
            const uint32_t o = atomicCAS(best, f, e);   // fails only where a better one came
            if (o == f) break;
            f = o;
          }
        }
        __syncthreads();
        for (uint32_t t0 = 0; t0 < m2; t0 += T) {
          uint32_t e[1] = {0u}, keep = 0;
          if (t0 + tid < m2) {
            e[0] = m.b[t0 + tid];
            const int r = (int)(e[0] >> 14);
            const P p = src.pt(e[0] & 0x3FFFu);
            const uint32_t f = m.tab[r * NB + blk_bucket<DT, NB>(s, p, r)];
            keep = f == e[0] || blk_key<DT>(p, r) < blk_key<DT>(src.pt(f & 0x3FFFu), r);
          }
          blk_append(m.a, &m.n[3], keep, e);
        }
        __syncthreads();
        m2 = m.n[3];
        for (uint32_t t = tid; t < m2; t += T) m.b[t] = m.a[t];
      }
      uint32_t N2 = 2;
      while (N2 < m2) N2 <<= 1;
      for (uint32_t t = m2 + tid; t < N2; t += T) m.b[t] = 0xFFFFu;
      __syncthreads();
      for (uint32_t k = 2; k <= N2; k <<= 1) {
        for (uint32_t d = k >> 1; d > 0; d >>= 1) {
          for (uint32_t i = tid; i < N2 / 2; i += T) {
            const uint32_t lo = 2 * i - (i & (d - 1)), hi = lo + d;
            const uint32_t x = m.b[lo], y = m.b[hi];
            bool gt;                               // x after y
            if (x == 0xFFFFu || y == 0xFFFFu || (x >> 14) != (y >> 14)) {
              gt = x > y;
            } else {
              const int r = (int)(x >> 14);
              const uint64_t kx = blk_key<DT>(src.pt(x & 0x3FFFu), r), ky = blk_key<DT>(src.pt(y & 0x3FFFu), r);
              gt = kx > ky || (kx == ky && x > y);
            }
            if (gt == ((lo & k) == 0)) { m.b[lo] = (uint16_t)y; m.b[hi] = (uint16_t)x; }
          }
          __syncthreads();
        }
      }
    }
    __syncthreads();
  }
  if (m2 <= kBlkWarpTail) {
    if (warp == 0) blk_tail<DT, 32>(m, src, m2);
  } else {
    blk_tail<DT, T>(m, src, m2);
  }
}

}  // namespace cch
