// k_set.cu -- the whole method (Sec. 2.1, steps 1-7) for a small set in one
// CTA, or in a cluster of four: the four extremes, the region test, and from the region points' list
// on the block steps of hull_block.cuh.  One launch, no workspace and no
// dependent kernels: a set of a few thousand points is nothing but latency in
// the streaming pipeline (nine launches, 80 us for 1000 points), and in a
// batch its regions would each hold an SM there.
//
// Measured (one GB300, us per call): one float64 set of 1000 / 3000 / 12000
// disk points 20 / 22 / 36 (the last two split over four CTAs; 29 / 54 in one)
// against 62 / 72 / 93 in the pipeline; 4096 float64 sets of 256 to 4096
// points 212 against 3092.  The exact tests of undecided
// points are the costly part: the extremes, which lie on the edges, are let
// past them (regions of 1000 points: 16k cycles before, 8k after), and one
// warp runs the last steps alone when few candidates are left (most sets).
//
// The points are read four times by coalesced loads (extremes, the rescan of
// the warps that hold one, regions, and the candidates); the set is at most
// 256 KB, so every read after the first hits L1 or L2.
#include <cooperative_groups.h>

#include "hull_block.cuh"

namespace cch {

// Size classes: sets of fewer than CAP points, T threads, NB buckets per
// region.  A class takes T threads for CAP / T <= 32 points each; smaller
// classes put more sets on an SM.
template <int C>
struct SetClass;
template <>
struct SetClass<0> { static constexpr int CAP = 1024, T = 128, NB = 128; };
template <>
struct SetClass<1> { static constexpr int CAP = 2048, T = 128, NB = 256; };
template <>
struct SetClass<2> { static constexpr int CAP = 4096, T = 256, NB = 512; };
template <>
struct SetClass<3> { static constexpr int CAP = 16384, T = 512, NB = 1280; };
// Split sets: there is an SM for every CTA, so more warps cost only their
// barriers (the sieve's lists, 512 -> 1024 threads, us per call: 2M annulus 147
// -> 135, 48,007 degenerate points 143 -> 127, 1M int32 square 56 -> 58).
template <>
struct SetClass<4> { static constexpr int CAP = 16384, T = 1024, NB = 1280; };
static_assert(SetClass<0>::CAP == kSetCap[0] && SetClass<1>::CAP == kSetCap[1] && SetClass<2>::CAP == kSetCap[2] &&
              SetClass<3>::CAP == kSetCap[3] && SetClass<4>::CAP == kSetCap[3], "the classes of set_class");

// Point c of the set, and the index it is reported as: its own, or that of the
// sieve's list (`map`).
template <int DT, bool LIST>
struct SetSrc {
  const Job& j;
  int64_t off;
  const uint32_t* map;
  __device__ __forceinline__ typename PT<DT>::T pt(uint32_t c) const { return input_point<typename PT<DT>::T>(j, off + c); }
  __device__ __forceinline__ int32_t out(uint32_t c) const { return LIST ? (int32_t)map[c] : (int32_t)c; }
};

// Order word of a leading word read as FP32, as a signed integer (-0.0 read as +0.0).
__device__ __forceinline__ int32_t lead_order(float f) { return (int32_t)(f32_order(__fadd_rn(f, 0.0f)) ^ 0x80000000u); }

// Whether p lies strictly outside edge k, exactly; and the first edge that has it
// outside (1..4, 0: none; int32: region_exact_i32).  Out of line: no other value of
// the caller lives across the tests' registers.
template <int DT>
__device__ __forceinline__ bool set_outside_in(const BlkSet<DT>& s, uint32_t k, const typename PT<DT>::T& p, uint32_t flags) {
  if (flags & (SF_DEGEN0 << k)) return false;
  const typename PT<DT>::T a = s.e[k], b = s.e[(k + 1) & 3u];
  if constexpr (DT == DT_F64) return orient_f64(a.x, a.y, b.x, b.y, p.x, p.y, (flags & SF_SMALL) != 0) < 0;
  else return orient_i32(a.x, a.y, b.x, b.y, p.x, p.y, (flags & SF_WIDE) != 0) < 0;
}
template <int DT>
__device__ __noinline__ bool set_outside(const BlkSet<DT>& s, uint32_t k, typename PT<DT>::T p, uint32_t flags) {
  return set_outside_in<DT>(s, k, p, flags);
}
static __device__ __noinline__ uint32_t set_region(const BlkSet<DT_F64>& s, double2 p, uint32_t flags) {
#pragma unroll 1
  for (uint32_t k = 0; k < 4u; k++)
    if (set_outside_in<DT_F64>(s, k, p, flags)) return k + 1;
  return 0;
}

// What k_set works on: the points of whole sets (items, or the one set); a
// single set's list from the sieve, w.sv_hdr->n points; or the lists of a
// batch's larger sets, which each CTA first gathers from its set's units.
enum : int { SET_WHOLE = 0, SET_LIST = 1, SET_BATCH = 2 };

// float32 vectors (DT_F64 with j.ys) are widened on load.  `beside`: the kernel
// before this one works on other sets of the same call, so this one starts
// beside it, and one of its CTAs waits for its end (all of them waiting would
// hold the SMs).
// SPLIT: a set is finished by a cluster of four CTAs: each does step 1 on all
// points, finds those of one region and does steps 4-7 on them; a region's
// chain ends in E1..E4, all of them vertices.  The sieve's lists lie close to
// the hull, so nearly all of their points reach the last steps (2300 points of a
// 20M disk: 57 us in one CTA, 45 of them from the sort on), and so do those of
// a circle.  It takes the SMs that a single set or a few leave idle (12,000
// points, one CTA / split / the pipeline: circle 166 / 59 / 134, beyond 2^60 1025
// / 218 / 225).
//
// 64 registers: what a thread can have where the shared memory of the smaller
// classes lets the SM fill up (72 and 80, which the exact tests would take:
// 4096 small float64 sets 306 us against 223).
template <int DT, int C, int MODE, bool SPLIT>
__global__ void __launch_bounds__(SetClass<C>::T, 1024 / SetClass<C>::T) k_set(Job j, const SetItem* items, Ws w, bool beside) {
  constexpr bool LIST = MODE == SET_LIST;
  static_assert(SPLIT || !LIST, "a single set's list is split");
  if (MODE != SET_WHOLE || !beside) griddep_enter();
  if constexpr (LIST) {
    if (!sieved(w)) return;
    griddep_release();                       // where it follows on this stream, the pipeline only leaves
  }
  if constexpr (MODE == SET_WHOLE) griddep_release();
  constexpr int CAP = SetClass<C>::CAP, T = SetClass<C>::T, NB = SetClass<C>::NB, NW = T / 32;
  using P = typename PT<DT>::T;
  using M = BlkSmem<DT, CAP, T, NB>;
  extern __shared__ __align__(16) unsigned char smem[];
  M& m = *reinterpret_cast<M*>(smem);
  __shared__ Lex red[NW][4];
  __shared__ uint32_t red_amin[NW];
  __shared__ int32_t wext[4][NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t part = SPLIT ? blockIdx.x & 3u : 0u;     // SPLIT: the CTA's region
  const uint32_t which = SPLIT ? blockIdx.x >> 2 : blockIdx.x;
  SetItem it = MODE == SET_WHOLE && items ? items[which] : SetItem{0, LIST ? (int32_t)w.sv_hdr->n : (int32_t)j.N, 0};
  if constexpr (MODE == SET_BATCH) {
    // gather the set's list (SPLIT: every CTA of the cluster, the same words);
    // a list of another size class, or too long a one (the pipeline's), is left
    const SieveSet sv = j.sv_sets[which];
    if (w.sv_hdr[which].mode == 0 || (j.sv_all && w.ctr[CT_SIEVE_NONE] != 0)) return;
    const uint32_t* cnt = w.sv_cnt + (size_t)sv.cta0 * kSvWarps;
    static_assert(kSvBatchUnits <= 4 * NB && kSvBatchUnits % T == 0, "the units' prefix fits the table");
    constexpr int PU = kSvBatchUnits / T;
    uint32_t c[PU], sum = 0, total;
#pragma unroll
    for (int q = 0; q < PU; q++) { const int u = tid * PU + q; c[q] = u < sv.nunit ? cnt[u] : 0u; sum += c[q]; }
    uint32_t pre = blk_excl_sum<T>(sum, m.w32[0], total);
    if (total > (uint32_t)kSetMax || (!SPLIT && (total < (uint32_t)SetClass<2>::CAP) != (C == 2))) return;
#pragma unroll
    for (int q = 0; q < PU; q++) { m.tab[tid * PU + q] = pre; pre += c[q]; }
    __syncthreads();
    P* lp = reinterpret_cast<P*>(w.cpts) + sv.off;       // j.pts is w.cpts
    const P* in = reinterpret_cast<const P*>(w.sv_in) + sv.off;
    for (uint32_t p = tid; p < total; p += T) {
      uint32_t l = 0, h = kSvBatchUnits - 1;             // the last unit that starts at or before p
      while (l < h) {
        const uint32_t q = (l + h + 1) >> 1;
        if (m.tab[q] <= p) l = q; else h = q - 1;
      }
      const uint32_t g = w.valA[sv.off + (int64_t)l * sv.len + (p - m.tab[l])];
      lp[p] = in[g];
      w.cidx[sv.off + p] = g;
    }
    __syncthreads();
    it = SetItem{sv.off, (int32_t)total, j.sets[which].id};
    if (tid == 0 && part == 0) {
      w.ctl[which].status = ST_SIEVED;
      if (atomicAdd(w.ctr + CT_SIEVE_SETS, 1u) + 1u == (uint32_t)j.nsets) w.ctr[CT_SIEVED] = 1u;
    }
  }
  const int n = it.n;
  int32_t* out_idx = j.out_idx + it.off;
  int32_t* out_count = j.out_counts + it.id;
  if (n == 0) {
    if (tid == 0) *out_count = 0;
    if (MODE == SET_WHOLE && beside && blockIdx.x == 0) griddep_enter();
    return;
  }
  const SetSrc<DT, MODE != SET_WHOLE> src{j, it.off, MODE == SET_BATCH ? w.cidx + it.off : w.cidx};
  for (int i = tid; i < 4 * NB; i += T) { m.tab[i] = 0xFFFFFFFFu; m.cnt[i] = 0u; }
  if (tid < 4) m.n[tid] = 0;
  if (tid == 0) m.s2 = 0;

  // ---- step 1: extremes of the leading words first (float64: the top word
  // read as FP32, in the order of a1's filter; int32: the coordinate), then
  // the exact lexicographic keys in the warps that reach one of the four
  bool rare, tiny = false;
  int32_t bnd[4];                          // the set's leading-word bounds
  uint32_t amin = 0x7FFFFFFFu;
  if constexpr (DT == DT_F64) {
    const float inf = __int_as_float(0x7F800000);
    float mnx = inf, mny = inf, mxx = -inf, mxy = -inf, tmn = inf;
#pragma unroll 4
    for (int i = tid; i < n; i += T) {
      const P p = src.pt(i);
      const float fx = __int_as_float(__double2hiint(p.x)), fy = __int_as_float(__double2hiint(p.y));
      tmn = fmin_nan(tmn, fmin_nan(fabsf(fx), fabsf(fy)));
      mnx = fmin_nan(mnx, fx); mny = fmin_nan(mny, fy);
      mxx = fmax_nan(mxx, fx); mxy = fmax_nan(mxy, fy);
    }
    // warp and CTA bounds as signed order words (-0.0 read as +0.0); a NaN
    // anywhere sends every warp to the exact keys
    const float v[4] = {mnx, mny, -mxx, -mxy};
    int32_t o[4];
    bool nan = false;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      nan |= v[k] != v[k];
      o[k] = lead_order(v[k]);
      const int32_t w = __reduce_min_sync(0xFFFFFFFFu, o[k]);
      if (lane == 0) wext[k][warp] = w;
    }
    const bool anynan = __syncthreads_or(nan) != 0;
    rare = anynan;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      int32_t b = wext[k][0];
#pragma unroll
      for (int q = 1; q < NW; q++) b = min(b, wext[k][q]);
      rare |= o[k] == b;
      bnd[k] = anynan ? 0x7FFFFFFF : b;
    }
    tiny = !(tmn >= kTinyTopF);            // zeros and tiny magnitudes: the domain check
    rare |= tiny;
  } else {
    int mnx = 0x7FFFFFFF, mny = 0x7FFFFFFF, mxx = (int)0x80000000, mxy = (int)0x80000000;
#pragma unroll 4
    for (int i = tid; i < n; i += T) {
      const P p = src.pt(i);
      mnx = min(mnx, p.x); mny = min(mny, p.y); mxx = max(mxx, p.x); mxy = max(mxy, p.y);
    }
    const int32_t o[4] = {mnx, mny, ~mxx, ~mxy};
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const int32_t w = __reduce_min_sync(0xFFFFFFFFu, o[k]);
      if (lane == 0) wext[k][warp] = w;
    }
    __syncthreads();
    rare = false;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      int32_t b = wext[k][0];
#pragma unroll
      for (int q = 1; q < NW; q++) b = min(b, wext[k][q]);
      rare |= o[k] == b;
      bnd[k] = b;
    }
  }
  {
    Lex best[4];
#pragma unroll
    for (int k = 0; k < 4; k++) { best[k].k1 = ~0ull; best[k].k2 = ~0ull; best[k].idx = 0xFFFFFFFFu; }
    if (__any_sync(0xFFFFFFFFu, rare)) {
      // only a point that reaches a bound can be an extreme: find those with
      // the loads in flight together, then take their exact keys
      uint32_t hit = 0;
#pragma unroll 4
      for (int i = tid, k = 0; i < n; i += T, k++) {
        const P p = src.pt(i);
        bool reach;
        if constexpr (DT == DT_F64) {
          const float fx = __fadd_rn(__int_as_float(__double2hiint(p.x)), 0.0f);
          const float fy = __fadd_rn(__int_as_float(__double2hiint(p.y)), 0.0f);
          reach = lead_order(fx) <= bnd[0] || lead_order(fy) <= bnd[1] || lead_order(-fx) <= bnd[2] ||
                  lead_order(-fy) <= bnd[3];
        } else {
          reach = p.x <= bnd[0] || p.y <= bnd[1] || ~p.x <= bnd[2] || ~p.y <= bnd[3];
        }
        hit |= (uint32_t)reach << k;
      }
      while (hit) {
        const int i = tid + (__ffs(hit) - 1) * T;
        hit &= hit - 1;
        uint32_t xh, xl, yh, yl, dummy = 0;
        a1_words<DT>(src.pt(i), xh, xl, yh, yl, dummy);
        a1_update<DT>(xh, xl, yh, yl, (uint32_t)i, best);
      }
      if (tiny) {
#pragma unroll 4
        for (int i = tid; i < n; i += T) {
          uint32_t xh, xl, yh, yl;
          a1_words<DT>(src.pt(i), xh, xl, yh, yl, amin);
        }
      }
#pragma unroll
      for (int k = 0; k < 4; k++) best[k] = lex_warp_min(best[k]);
      amin = __reduce_min_sync(0xFFFFFFFFu, amin);
    }
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < 4; k++) red[warp][k] = best[k];
      red_amin[warp] = amin;
    }
  }
  __syncthreads();
  // ---- set-up by one warp: lane k < 4 owns extreme, edge and region k
  BlkSet<DT>& s = m.s;
  if (warp == 0) {
    Lex best[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
      Lex v{~0ull, ~0ull, 0xFFFFFFFFu};
      if (lane < NW) v = red[lane][k];
      best[k] = lex_warp_min(v);
    }
    amin = __reduce_min_sync(0xFFFFFFFFu, lane < NW ? red_amin[lane] : 0x7FFFFFFFu);
    const int k1 = (lane + 1) & 3;
    const uint32_t myidx = lane == 0 ? best[0].idx : lane == 1 ? best[1].idx : lane == 2 ? best[2].idx : best[3].idx;
    if (lane < 4) {
      const P p = src.pt(myidx);
      s.e[lane] = p;
      s.ex[lane] = (double)p.x;
      s.ey[lane] = (double)p.y;
      s.eidx[lane] = myidx;
    }
    __syncwarp();
    uint32_t flags = 0;
    int st = 0;
    const double xm = fmax(fabs(s.ex[0]), fabs(s.ex[2])), ym = fmax(fabs(s.ey[1]), fabs(s.ey[3]));
    bool small = true;
    if constexpr (DT == DT_F64) {
      // NaN, Inf and huge values sort beyond every finite value, so they are
      // among the extremes; tiny nonzero values were folded into amin
      for (int k = 0; k < 4; k++) {
        const uint32_t bx = f64_bad((uint64_t)__double_as_longlong(s.ex[k]));
        const uint32_t by = f64_bad((uint64_t)__double_as_longlong(s.ey[k]));
        if (bx == 1u || by == 1u) st = ST_NONFINITE;
        else if ((bx | by) && st == 0) st = ST_RANGE;
      }
      if (st == 0 && amin < ((1023u - 400u) << 20)) st = ST_RANGE;
      small = xm <= 1152921504606846976.0 && ym <= 1152921504606846976.0;   // 2^60
      if (small) flags |= SF_SMALL;
    } else {
      if (s.ex[2] - s.ex[0] >= 2147483648.0 || s.ey[3] - s.ey[1] >= 2147483648.0) flags |= SF_WIDE;
    }
#pragma unroll
    for (int k = 0; k < 4; k++)
      if (best[k].idx == best[(k + 1) & 3].idx) flags |= SF_DEGEN0 << k;
    if (lane == 0) {
      s.flags = flags;
      s.status = st;
      s.down = small ? 0u : ((uint32_t)__double2hiint(fmax(xm, ym)) & 0x7FF00000u) - (1023u << 20);
    }
    __syncwarp();
    if (lane < 4 && st == 0) {
      edge_filter(s.ex[lane], s.ey[lane], s.ex[k1], s.ey[k1], xm, ym, small, s.fA[lane], s.fB[lane], s.fC[lane],
                  s.fE[lane]);
      blk_map<DT, NB>(s, lane);
    }
  }
  __syncthreads();
  if (s.status != 0) {
    if (tid == 0 && part == 0) *out_count = s.status;
    if (MODE == SET_WHOLE && beside && blockIdx.x == 0) griddep_enter();
    return;
  }
  // ---- steps 2-3: the first edge that has the point strictly outside is its
  // region; the FP32 filter decides where it can (round1.cuh), then the exact
  // test.  Region points are listed and enter the dominance table.  SPLIT: only
  // whether it is the CTA's region matters: the CTA's own edge first, and the
  // earlier ones only for a point outside it.
  {
    float fA[4], fB[4], fC[4], fE[4];
#pragma unroll
    for (int k = 0; k < 4; k++) { fA[k] = s.fA[k]; fB[k] = -s.fB[k]; fC[k] = s.fC[k]; fE[k] = s.fE[k]; }
    const uint32_t flags = s.flags;
    uint32_t eidx[4];
#pragma unroll
    for (int k = 0; k < 4; k++) eidx[k] = s.eidx[k];
    for (int i0 = 0; i0 < n; i0 += 4 * T) {
      uint32_t rr = 0, und = 0;          // regions (4 bits each) and undecided points of the thread's four
      {
        P p[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
          const int i = i0 + u * T + tid;
          if (i < n) p[u] = src.pt(i);
        }
#pragma unroll
        for (int u = 0; u < 4; u++) {
          if (i0 + u * T + tid < n) {
            float X, Y;
            f32_view<DT>(p[u], X, Y);
            uint32_t r = 0;
#pragma unroll
            for (int k = 3; k >= 0; k--) {
              const float d = __fmaf_rn(fA[k], Y, __fmaf_rn(fB[k], X, fC[k]));
              r = !(d > fE[k]) ? (d < -fE[k] ? k + 1 : 8) : r;
            }
            if (r == 8) und |= 1u << u;
            else rr |= r << (4 * u);
          }
        }
      }
      // the few undecided points, read again (no other value lives across the
      // exact test); the extremes themselves lie on the edges: no region
      while (und) {
        const int u = __ffs(und) - 1;
        und &= und - 1;
        const uint32_t i = (uint32_t)(i0 + u * T + tid);
        if (i == eidx[0] || i == eidx[1] || i == eidx[2] || i == eidx[3]) continue;
        const P p = src.pt(i);
        uint32_t r = 0;
        if constexpr (!SPLIT) {
          if constexpr (DT == DT_F64) r = set_region(s, p, flags);
          else r = (uint32_t)region_exact_i32(p.x, p.y, s.ex, s.ey, flags);
        } else if (set_outside<DT>(s, part, p, flags)) {
          for (uint32_t k = 0; k < part && r == 0; k++)
            if (set_outside<DT>(s, k, p, flags)) r = k + 1;
          if (r == 0) r = part + 1;
        }
        rr |= r << (4 * u);
      }
      uint32_t e[4], take = 0;
#pragma unroll
      for (int u = 0; u < 4; u++) {
        const uint32_t i = (uint32_t)(i0 + u * T + tid), r = (rr >> (4 * u)) & 7u;
        e[u] = ((r - 1u) << 14) | i;
        if (SPLIT ? r == part + 1u : r != 0) {
          const P p = src.pt(i);
          atomicMin(&m.tab[(r - 1) * NB + blk_bucket<DT, NB>(s, p, (int)r - 1)],
                    blk_word<DT>(blk_spa<DT>(p, (int)r - 1)));
          take |= 1u << u;
        }
      }
      blk_append(m.a, &m.n[0], take, e);
    }
  }
  __syncthreads();
  uint32_t at = 0;                             // first output slot of the CTA's vertices
  if constexpr (SPLIT) {
    const uint32_t flags = s.flags, all = SF_DEGEN0 * 15u, mine = SF_DEGEN0 << part;
    __syncthreads();
    if (tid == 0) {
      if ((flags & all) != all) s.flags = flags | (all & ~mine);   // this region's chain alone
      m.close = s.eidx[(part + 1u) & 3u];
      m.hn = 0;
      m.hb = 0;
    }
    __syncthreads();
    // a region between coincident extremes has no chain; all coincident: the
    // first CTA's single point
    if (!(flags & mine) || ((flags & all) == all && part == 0)) blk_finish<DT, CAP, T, NB>(m, src);
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    uint32_t tot = 0;
#pragma unroll
    for (uint32_t q = 0; q < 4; q++) {
      const uint32_t c = *cl.map_shared_rank(&m.hn, q);
      at += q < part ? c : 0u;
      tot += c;
    }
    cl.sync();                                 // nobody leaves while its count is read
    if (tid == 0 && part == 0) *out_count = (int32_t)tot;
  } else {
    if (tid == 0) {
      int k = 0;                               // the first region with a chain
      while (k < 3 && (s.flags & (SF_DEGEN0 << k))) k++;
      m.close = s.eidx[k];
    }
    blk_finish<DT, CAP, T, NB>(m, src);
    __syncthreads();
    if (tid == 0) *out_count = (int32_t)m.hn;
  }
  const uint16_t* h = m.hb ? m.b : m.a;
  for (uint32_t t = tid; t < m.hn; t += T) out_idx[at + t] = src.out(h[t] & ~kPin);
  if (MODE == SET_WHOLE && beside && blockIdx.x == 0) griddep_enter();
}

template <int DT, int C, int MODE, bool SPLIT>
static void launch_set_c(const Job& j, const SetItem* items, const Ws& w, int count, bool beside, cudaStream_t st) {
  constexpr size_t sm = sizeof(BlkSmem<DT, SetClass<C>::CAP, SetClass<C>::T, SetClass<C>::NB>);
  static bool once = [] {
    cudaFuncSetAttribute(k_set<DT, C, MODE, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    return true;
  }();
  (void)once;
  launch_pdl_cluster(k_set<DT, C, MODE, SPLIT>, SPLIT ? 4 * count : count, SetClass<C>::T, SPLIT ? 4 : 1, sm, st, j, items,
                     w, beside);
}

template <int DT>
static void launch_set_t(const Job& j, int cls, const SetItem* items, int count, bool split, bool beside,
                         cudaStream_t st) {
  if (split) launch_set_c<DT, 4, SET_WHOLE, true>(j, items, Ws{}, count, beside, st);
  else if (cls == 0) launch_set_c<DT, 0, SET_WHOLE, false>(j, items, Ws{}, count, beside, st);
  else if (cls == 1) launch_set_c<DT, 1, SET_WHOLE, false>(j, items, Ws{}, count, beside, st);
  else if (cls == 2) launch_set_c<DT, 2, SET_WHOLE, false>(j, items, Ws{}, count, beside, st);
  else launch_set_c<DT, 3, SET_WHOLE, false>(j, items, Ws{}, count, beside, st);
}

int launch_set(const Job& j, int cls, const SetItem* items, int count, bool split, bool beside, cudaStream_t st) {
  if (count == 0) return 0;
  if (j.dtype == DT_I32) launch_set_t<DT_I32>(j, cls, items, count, split, beside, st);
  else launch_set_t<DT_F64>(j, cls, items, count, split, beside, st);
  return 1;
}

template <int DT>
static int launch_set_list_t(const Job& l, const Ws& w, int sms, cudaStream_t st) {
  if (!l.sv_sets) {
    launch_set_c<DT, 4, SET_LIST, true>(l, nullptr, w, 1, false, st);
    return 1;
  }
  if (l.nsets <= sms / 4) {
    launch_set_c<DT, 4, SET_BATCH, true>(l, nullptr, w, l.nsets, false, st);
    return 1;
  }
  launch_set_c<DT, 2, SET_BATCH, false>(l, nullptr, w, l.nsets, false, st);
  launch_set_c<DT, 3, SET_BATCH, false>(l, nullptr, w, l.nsets, false, st);
  return 2;
}

int launch_set_list(const Job& j, const Ws& w, int sms, cudaStream_t st) {
  Job l = j;
  l.pts = w.cpts;          // float32 vectors are listed widened
  l.ys = nullptr;
  Ws v = w;
  v.sv_in = j.pts;
  return j.dtype == DT_I32 ? launch_set_list_t<DT_I32>(l, v, sms, st) : launch_set_list_t<DT_F64>(l, v, sms, st);
}

}  // namespace cch
