// Radius search and k-NN over a CGA (the Eq. 8 set generalised): every
// stored voxel within a squared integer distance r2 of each query voxel in
// ascending CGA index, or the k least (distance^2, key) in ascending order.
//   k_radius_count  one warp per query: the slabs whose x lies within the
//                   radius (the x directory gives them) are shared 32 at a time
//                   among the lanes; a lane walks its slab's columns inside the
//                   circle left for y and counts each column's voxels in reach:
//                   short columns voxel by voxel, long ones by two searches
//   k_scan_*        exclusive prefix of the counts (64-bit offsets)
//   k_radius_fill   the same walk; per group of 32 slabs a warp scan of the
//                   lanes' counts places every slab's voxels, so the output
//                   is in (x, y, z) = CGA order without sorting
// The walks are bound by load latency and integer instructions (DRAM below 2% of
// its bandwidth), so a radius below 2^31 (r^2 in voxels) runs in 32-bit
// arithmetic: every coordinate difference inside the windows is at most r.
// Measured, 1M queries of 10 cm in the 0.94M-voxel LiDAR world (21M results),
// count and fill with the order of the queries: 5.8 -> 3.2 ms (64-bit walks, the
// slabs by search, the fill walking every slab twice; 3.9 ms before the grid was
// cut to one wave and the hits staged for whole-sector stores).  k-NN of the
// same queries: k = 8 6.9 -> 5.7 ms, k = 400 (100k queries) 16.0 -> 11.4 ms with
// pairs of one 64-bit word.  Warps taking their block's next query when free: radius
// 3.0 ms, k = 8 5.3, k = 400 11.1; bound by instruction issue and load latency.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "k_common.cuh"

// Blocks per SM the search kernels are compiled for (their register budgets;
// measured on GB300: k-NN 4 / 5 / 6 blocks 6.26 / 5.69 / 6.06 ms; radius 5 / 6
// blocks 3.98 / 3.82 ms, 7 spill and take 5.9).
#ifndef CGA_KNN_BLOCKS
#define CGA_KNN_BLOCKS 5
#endif
#ifndef CGA_RADIUS_BLOCKS
#define CGA_RADIUS_BLOCKS 6
#endif

namespace libcga {

namespace {

// Largest s with s * s <= v (v < 2^63).  Below 2^46 a single-precision
// estimate is within 2 of the root (the rounding of v to float moves the
// root by at most a quarter, sqrtf's own rounding by at most half a unit of
// a number below 2^23), so two exact integer steps at most fix it; the rare
// larger arguments take the double-precision estimate, which GB300 runs at a
// small fraction of the single-precision rate.
__device__ __forceinline__ unsigned long long isqrt_u64(unsigned long long v) {
  unsigned long long s = v < (1ull << 46) ? (unsigned long long)sqrtf((float)v)
                                          : (unsigned long long)sqrt((double)v);
  while (s > 0 && s * s > v) --s;
  while ((s + 1) * (s + 1) <= v) ++s;
  return s;
}

// The same for a 32-bit argument, in 32-bit arithmetic.
__device__ __forceinline__ uint32_t isqrt_u32(uint32_t v) {
  uint32_t s = min((uint32_t)sqrtf((float)v), 65535u);
  if (s * s > v) --s;
  if (s < 65535u && (s + 1) * (s + 1) <= v) ++s;
  return s;
}
__device__ __forceinline__ uint32_t isqrt_of(uint32_t v) { return isqrt_u32(v); }
__device__ __forceinline__ unsigned long long isqrt_of(unsigned long long v) { return isqrt_u64(v); }

// |v - q| of a stored coordinate and a query coordinate (clamped to
// +-2^30, so the difference fits 31 bits).
__device__ __forceinline__ uint32_t absdiff32(uint32_t v, int q) {
  const int d = (int)v - q;
  return (uint32_t)(d < 0 ? -d : d);
}

// The grid coordinates [lo, hi] within r of q on one axis, cut to [0, top] (in
// 64 bits where the reach may exceed 2^31).  False when empty.
__device__ __forceinline__ bool axis_window(int q, unsigned long long r, int top, int& lo, int& hi) {
  const long long l = (long long)q - (long long)r, h = (long long)q + (long long)r;
  if (h < 0 || l > top) return false;
  lo = (int)max(l, 0ll);
  hi = (int)min(h, (long long)top);
  return true;
}
__device__ __forceinline__ bool axis_window(int q, uint32_t r, int top, int& lo, int& hi) {
  lo = max(q - (int)r, 0);  // |q| <= 2^30 and r < 2^16: no overflow
  hi = min(q + (int)r, top);
  return lo <= hi;
}


struct RQuery {
  int x, y, z;  // query voxel (clamped only to +-2^30)
  bool valid;
};

__device__ __forceinline__ RQuery radius_query(const SearchSeg& sg, uint32_t j) {
  const float* p = sg.q + 3 * (size_t)j;
  const float px = __ldg(p), py = __ldg(p + 1), pz = __ldg(p + 2);
  RQuery q;
  q.valid = isfinite(px) && isfinite(py) && isfinite(pz);
  q.x = q.valid ? (int)quantize_query(px, sg.scale, sg.off[0]) : 0;
  q.y = q.valid ? (int)quantize_query(py, sg.scale, sg.off[1]) : 0;
  q.z = q.valid ? (int)quantize_query(pz, sg.scale, sg.off[2]) : 0;
  return q;
}

// Column c's voxel range [zs, ze) and z range [zlo, zhi]: one load from the
// column table when there is one, else the range is taken as the whole axis
// (so every shortcut below falls back to a search).
__device__ __forceinline__ void column_of(const Levels& a, const uint4* ctab, uint32_t c,
                                          uint32_t& zs, uint32_t& ze, uint32_t& zlo,
                                          uint32_t& zhi) {
  if (ctab != nullptr) {
    const uint4 e = __ldg(ctab + c);
    zs = e.x;
    ze = e.y;
    zlo = e.z & 0xffffu;
    zhi = e.z >> 16;
  } else {
    zs = __ldg(a.ptr1 + c);
    ze = __ldg(a.ptr1 + c + 1);
    zlo = 0;
    zhi = 0xffffu;
  }
}

// Slabs [s0, s1) of a whose x lies within r of the query's.
template <typename D>
__device__ __forceinline__ void radius_slabs(const SearchSeg& sg, uint32_t h, const RQuery& q, D r,
                                             uint32_t& s0, uint32_t& s1) {
  s0 = s1 = 0;
  int lo, hi;
  if (!q.valid || h == 0 || !axis_window(q.x, r, (1 << sg.a.bits) - 1, lo, hi)) return;
  if (sg.xdir != nullptr) {
    s0 = __ldg(sg.xdir + lo);
    s1 = __ldg(sg.xdir + hi + 1);
  } else {
    s0 = lower_bound_u16(sg.a.idx2, 0, h, (uint32_t)lo);
    s1 = lower_bound_u16(sg.a.idx2, s0, h, (uint32_t)hi + 1);
  }
}

// Up to this many voxels of a column are measured one by one (two 64-byte
// sectors at most); a longer column's reach comes from a root and two searches.
constexpr uint32_t kShortColumn = 4;

// The voxels of one slab within the radius, in (y, z) order: emit(p, d2) for each
// (of a long column, while more() says so).  Returns their number.  Only the slab's x
// lies inside the window, so every difference here is at most r (D = uint32_t: r2 < 2^31).
template <typename D, typename F, typename M>
__device__ __forceinline__ uint32_t radius_slab(const SearchSeg& sg, uint32_t slab, const RQuery& q,
                                                D r2, F emit, M more) {
  const Levels& a = sg.a;
  const int top = (1 << a.bits) - 1;
  const D dx = absdiff32(__ldg(a.idx2 + slab), q.x);
  const uint32_t ys = __ldg(a.ptr2 + slab), ye = __ldg(a.ptr2 + slab + 1);
  const D dx2 = dx * dx;
  if (dx2 > r2) return 0;
  int ylo, yhi;
  if (!axis_window(q.y, isqrt_of(r2 - dx2), top, ylo, yhi)) return 0;
  uint32_t n = 0;
  for (uint32_t c = lower_bound_u16(a.idx1, ys, ye, (uint32_t)ylo); c < ye; ++c) {
    const uint32_t y = __ldg(a.idx1 + c);
    if ((int)y > yhi) break;
    const D dy = absdiff32(y, q.y);
    const D dxy = dx2 + dy * dy, rem = r2 - dxy;
    uint32_t zs, ze, clo, chi;
    column_of(a, sg.ctab, c, zs, ze, clo, chi);
    if (ze - zs <= kShortColumn) {
      for (uint32_t p = zs; p < ze; ++p) {
        const uint32_t e = absdiff32(__ldg(a.idx0 + p), q.z);
        // (a difference beyond 65535 would wrap its 32-bit square)
        const D d = (D)e * e;
        if ((sizeof(D) == 8 || e <= 65535u) && d <= rem) {
          emit(p, dxy + d);
          ++n;
        }
      }
      continue;
    }
    int zlo, zhi;
    if (!axis_window(q.z, isqrt_of(rem), top, zlo, zhi)) continue;
    if ((uint32_t)zhi < clo || (uint32_t)zlo > chi) continue;
    const uint32_t p0 = (uint32_t)zlo <= clo ? zs : lower_bound_u16(a.idx0, zs, ze, (uint32_t)zlo);
    const uint32_t p1 =
        (uint32_t)zhi >= chi ? ze : lower_bound_u16(a.idx0, p0, ze, (uint32_t)zhi + 1);
    for (uint32_t p = p0; p < p1 && more(); ++p) {
      const D dz = absdiff32(__ldg(a.idx0 + p), q.z);
      emit(p, dxy + dz * dz);
    }
    n += p1 - p0;
  }
  return n;
}

// Query of slot `slot`: the slot itself, or the index in the low 32 bits of
// the Morton-ordered key when an order is given (neighbouring warps then
// search neighbouring space and share the cache).
__device__ __forceinline__ uint32_t slot_query(const unsigned long long* order, uint32_t slot) {
  return order != nullptr ? (uint32_t)__ldg(order + slot) : slot;
}

// r2 and its integer root r.
template <typename D>
__global__ void __launch_bounds__(256, CGA_RADIUS_BLOCKS)
    k_radius_count(SearchSeg sg, D r2, D r, const unsigned long long* __restrict__ order,
                   unsigned long long* counts) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t h = (uint32_t)sg.a.hdr->cnt[2];
  __shared__ uint32_t s_next;
  open_slots<256 / 32>(&s_next);
  for (uint32_t turn = threadIdx.x >> 5;; turn = next_turn(&s_next)) {
    const uint32_t sl = slot_of_turn<256 / 32>(turn);
    if (sl >= sg.m) break;
    const uint32_t j = slot_query(order, sl);
    const RQuery q = radius_query(sg, j);
    uint32_t s0, s1;
    radius_slabs<D>(sg, h, q, r, s0, s1);
    uint32_t n = 0;  // at most the CGA's voxels: below 2^30
    for (uint32_t s = s0 + lane; s < s1; s += 32) {
      n += radius_slab<D>(sg, s, q, r2, [](uint32_t, D) {}, [] { return false; });
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) counts[j] = n;
  }
}

// Hits of a lane's slab kept in shared memory until their place is known.  A lane with
// more of them walks its slab again and writes them then; the first walk only counts the
// rest of its long columns (looking at every voxel twice took 100 queries of 17 voxels
// in a world of 300k LiDAR points, b = 10, 322 us, 301 so).
constexpr uint32_t kRadiusKeep = 6;

template <typename D>
__global__ void __launch_bounds__(256, CGA_RADIUS_BLOCKS)
    k_radius_fill(SearchSeg sg, D r2, D r, const unsigned long long* __restrict__ order,
                  const unsigned long long* __restrict__ offsets, uint32_t* idx,
                  unsigned long long* d2) {
  __shared__ uint32_t s_p[kRadiusKeep][256];
  __shared__ D s_d[kRadiusKeep][256];
  // the group's hits in order, for whole-sector stores
  __shared__ uint32_t s_op[8][32 * kRadiusKeep];
  __shared__ D s_od[8][32 * kRadiusKeep];
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  const uint32_t h = (uint32_t)sg.a.hdr->cnt[2];
  __shared__ uint32_t s_next;
  open_slots<256 / 32>(&s_next);
  for (uint32_t turn = tid >> 5;; turn = next_turn(&s_next)) {
    const uint32_t sl = slot_of_turn<256 / 32>(turn);
    if (sl >= sg.m) break;
    const uint32_t j = slot_query(order, sl);
    const RQuery q = radius_query(sg, j);
    uint32_t s0, s1;
    radius_slabs<D>(sg, h, q, r, s0, s1);
    unsigned long long base = __ldg(offsets + j);
    for (uint32_t g = s0; g < s1; g += 32) {
      const uint32_t s = g + lane;
      uint32_t n = 0, kept = 0;
      if (s < s1) {
        n = radius_slab<D>(sg, s, q, r2, [&](uint32_t p, D d) {
          if (kept < kRadiusKeep) {
            s_p[kept][tid] = p;
            s_d[kept][tid] = d;
          }
          ++kept;
        }, [&] { return kept < kRadiusKeep; });
      }
      const uint32_t inc = warp_incl_scan(n);
      const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
      if (total == 0) continue;
      if (__all_sync(0xffffffffu, n <= kRadiusKeep)) {
        uint32_t* op = s_op[tid >> 5];
        D* od = s_od[tid >> 5];
        for (uint32_t e = 0; e < n; ++e) {
          op[inc - n + e] = s_p[e][tid];
          od[inc - n + e] = s_d[e][tid];
        }
        __syncwarp();
        for (uint32_t e = lane; e < total; e += 32) {
          idx[base + e] = op[e];
          d2[base + e] = od[e];
        }
        __syncwarp();
      } else if (n > 0) {
        // a lane with more hits than it keeps: once more, straight to their places
        unsigned long long at = base + inc - n;
        radius_slab<D>(sg, s, q, r2, [&](uint32_t p, D d) {
          idx[at] = p;
          d2[at] = d;
          ++at;
        }, [] { return true; });
      }
      base += total;
    }
  }
}

// Exclusive scan of v[0, m) in place, v[m] = total: B blocks, each owning a
// contiguous chunk; block totals are scanned by one block, then each chunk
// is rescanned with its prefix.
__global__ void k_scan_totals(const unsigned long long* v, uint64_t m, uint64_t chunk,
                              unsigned long long* totals) {
  __shared__ unsigned long long s_warp[kWarps];
  const uint64_t lo = blockIdx.x * chunk, hi = min(lo + chunk, m);
  unsigned long long t = 0;
  for (uint64_t i = lo + threadIdx.x; i < hi; i += kThreads) t += v[i];
  unsigned long long tot;
  block_excl_scan(t, tot, s_warp);
  if (threadIdx.x == 0) totals[blockIdx.x] = tot;
}

// B <= 1024 totals, four a thread.
__global__ void __launch_bounds__(kThreads) k_scan_top(unsigned long long* totals, uint32_t B) {
  __shared__ unsigned long long s_warp[kWarps];
  unsigned long long t[4], sum = 0, tot = 0;
#pragma unroll
  for (uint32_t i = 0; i < 4; ++i) {
    const uint32_t b = 4 * threadIdx.x + i;
    t[i] = b < B ? totals[b] : 0ull;
    sum += t[i];
  }
  unsigned long long run = block_excl_scan(sum, tot, s_warp);
#pragma unroll
  for (uint32_t i = 0; i < 4; ++i) {
    const uint32_t b = 4 * threadIdx.x + i;
    if (b < B) totals[b] = run;
    run += t[i];
  }
  if (threadIdx.x == 0) totals[B] = tot;
}

__global__ void k_scan_apply(unsigned long long* v, uint64_t m, uint64_t chunk,
                             const unsigned long long* totals, uint32_t B) {
  __shared__ unsigned long long s_warp[kWarps];
  const uint64_t lo = blockIdx.x * chunk, hi = min(lo + chunk, m);
  unsigned long long run = totals[blockIdx.x];
  for (uint64_t b0 = lo; b0 < hi; b0 += kThreads) {
    const uint64_t i = b0 + threadIdx.x;
    const unsigned long long x = i < hi ? v[i] : 0ull;
    unsigned long long tot;
    const unsigned long long ex = block_excl_scan(x, tot, s_warp);
    if (i < hi) v[i] = run + ex;
    run += tot;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) v[m] = totals[B];
}

// ---- k nearest -------------------------------------------------------------
// The search collects (distance^2, index) pairs.  The CGA index of a voxel
// rises with its key, so this order is (distance^2, key) order.
//
// Narrow form (the first launch): pairs as one 64-bit word, the squared distance
// (below 2^32 - 1) above the index, so that a comparison is one, a shuffle two,
// a list entry 8 bytes, and the walk runs in 32-bit arithmetic; voxels farther
// away are passed over.  A query that then has fewer than min(k, u) neighbours
// (its k-th lies 65536 or more voxels off) is answered by a second launch in the
// wide form, distances of 64 bits next to the index.
template <bool NARROW>
struct Pair;
template <>
struct Pair<true> {
  using D = uint32_t;
  static constexpr D kFar = 0xfffffffeu;  // the largest distance the form holds
  unsigned long long v;
  __device__ __forceinline__ static Pair none() { return Pair{~0ull}; }
  __device__ __forceinline__ static Pair of(D d, uint32_t i) {
    return Pair{(unsigned long long)d << 32 | i};
  }
  __device__ __forceinline__ bool less(const Pair& o) const { return v < o.v; }
  __device__ __forceinline__ D bound() const { return min((D)(v >> 32), kFar); }
  __device__ __forceinline__ Pair shfl(uint32_t src) const {
    return Pair{__shfl_sync(0xffffffffu, v, src)};
  }
  __device__ __forceinline__ Pair shfl_up1() const {
    return Pair{__shfl_up_sync(0xffffffffu, v, 1)};
  }
  __device__ __forceinline__ Pair shfl_xor(uint32_t m) const {
    return Pair{__shfl_xor_sync(0xffffffffu, v, m)};
  }
  __device__ __forceinline__ void write(uint32_t* idx, unsigned long long* d2, size_t at) const {
    idx[at] = (uint32_t)v;
    d2[at] = v == ~0ull ? ~0ull : v >> 32;
  }
  __device__ __forceinline__ static D square(uint32_t e) { return e > 65535u ? ~0u : e * e; }
  __device__ __forceinline__ static D plus(D a, D b) {
    const D s = a + b;
    return s < a ? ~0u : s;
  }
};
template <>
struct Pair<false> {
  using D = unsigned long long;
  static constexpr D kFar = ~0ull;
  unsigned long long d;
  uint32_t i;
  __device__ __forceinline__ static Pair none() { return Pair{~0ull, 0xffffffffu}; }
  __device__ __forceinline__ static Pair of(D d, uint32_t i) { return Pair{d, i}; }
  __device__ __forceinline__ bool less(const Pair& o) const {
    return d < o.d || (d == o.d && i < o.i);
  }
  __device__ __forceinline__ D bound() const { return d; }
  __device__ __forceinline__ Pair shfl(uint32_t src) const {
    return Pair{__shfl_sync(0xffffffffu, d, src), __shfl_sync(0xffffffffu, i, src)};
  }
  __device__ __forceinline__ Pair shfl_up1() const {
    return Pair{__shfl_up_sync(0xffffffffu, d, 1), __shfl_up_sync(0xffffffffu, i, 1)};
  }
  __device__ __forceinline__ Pair shfl_xor(uint32_t m) const {
    return Pair{__shfl_xor_sync(0xffffffffu, d, m), __shfl_xor_sync(0xffffffffu, i, m)};
  }
  __device__ __forceinline__ void write(uint32_t* idx, unsigned long long* d2, size_t at) const {
    idx[at] = i;
    d2[at] = d;
  }
  __device__ __forceinline__ static D square(uint32_t e) { return (D)e * e; }
  __device__ __forceinline__ static D plus(D a, D b) { return a + b; }
};

// One compare-exchange step of a bitonic network across the warp: the pair
// (lane, lane ^ j) is put in ascending order when `up`, descending otherwise.
template <typename P>
__device__ __forceinline__ void bitonic_step(P& p, uint32_t lane, uint32_t j, bool up) {
  const P o = p.shfl_xor(j);
  const bool keep_min = ((lane & j) == 0) == up;
  if (keep_min ? o.less(p) : p.less(o)) p = o;
}

// Above this many candidates in one step, one bitonic merge is cheaper than
// inserting them one by one.
constexpr int kKnnBatch = 8;
constexpr uint32_t kKnnLargeThreads = 128;  // 4 warps, each with its own buffer

// Candidate collection for k <= 32: the list in registers, lane i holding the
// i-th best; lanes >= k hold no pair.
template <bool NARROW>
struct RegList {
  using P = Pair<NARROW>;
  using D = typename P::D;
  P t;
  uint32_t k;

  __device__ __forceinline__ void init(uint32_t kk) {
    t = P::none();
    k = kk;
  }
  // One candidate (the same in every lane): it enters before the first entry
  // that is not below it, the entries after it move up one lane and the k-th
  // falls out.
  __device__ __forceinline__ void insert(const P& c, uint32_t lane) {
    const uint32_t pos = __popc(__ballot_sync(0xffffffffu, lane < k && t.less(c)));
    const P up = t.shfl_up1();
    if (lane >= pos && lane < k) t = lane == pos ? c : up;
  }
  // Every lane's candidate at once: the candidates are sorted by a bitonic
  // network, the lane-wise minimum of the list and the reversed candidates holds
  // the 32 least of both as a bitonic sequence, and a bitonic merge orders it.
  __device__ __forceinline__ void insert_all(P c, uint32_t lane) {
#pragma unroll
    for (uint32_t w = 2; w <= 32; w <<= 1) {
#pragma unroll
      for (uint32_t j = w >> 1; j > 0; j >>= 1) bitonic_step(c, lane, j, (lane & w) == 0);
    }
    const P r = c.shfl(31 - lane);
    if (r.less(t)) t = r;
#pragma unroll
    for (uint32_t j = 16; j > 0; j >>= 1) bitonic_step(t, lane, j, true);
    if (lane >= k) t = P::none();
  }
  // Offer each lane's candidate (if any); returns the new pruning bound.
  __device__ __forceinline__ D offer(bool has, D cd, uint32_t ci, uint32_t lane, D) {
    const P c = has ? P::of(cd, ci) : P::none();
    uint32_t pending = __ballot_sync(0xffffffffu, has);
    if (__popc(pending) > kKnnBatch) {
      insert_all(c, lane);
    } else {
      while (pending) {
        const uint32_t src = __ffs(pending) - 1;
        pending &= pending - 1;
        insert(c.shfl(src), lane);
      }
    }
    return t.shfl(k - 1).bound();
  }
  __device__ __forceinline__ void finish(uint32_t lane, size_t row, uint32_t* out_idx,
                                         unsigned long long* out_d2) {
    if (lane < k) t.write(out_idx, out_d2, row + lane);
  }
};

// The entries of a shared-memory buffer: words of the narrow form, or distances
// and indices apart.
template <bool NARROW>
struct PairBuf;
template <>
struct PairBuf<true> {
  static constexpr size_t kBytes = 8;
  unsigned long long* v;
  __device__ __forceinline__ void init(unsigned char* base, uint32_t wb, uint32_t, uint32_t cap) {
    v = reinterpret_cast<unsigned long long*>(base) + (size_t)wb * cap;
  }
  __device__ __forceinline__ Pair<true> get(uint32_t e) const { return Pair<true>{v[e]}; }
  __device__ __forceinline__ void set(uint32_t e, const Pair<true>& p) { v[e] = p.v; }
  __device__ __forceinline__ uint32_t dist(uint32_t e) const {
    return reinterpret_cast<const uint32_t*>(v)[2 * e + 1];
  }
};
template <>
struct PairBuf<false> {
  static constexpr size_t kBytes = 12;
  unsigned long long* d;
  uint32_t* ix;
  __device__ __forceinline__ void init(unsigned char* base, uint32_t wb, uint32_t warps,
                                       uint32_t cap) {
    d = reinterpret_cast<unsigned long long*>(base) + (size_t)wb * cap;
    ix = reinterpret_cast<uint32_t*>(base + (size_t)warps * cap * 8) + (size_t)wb * cap;
  }
  __device__ __forceinline__ Pair<false> get(uint32_t e) const { return Pair<false>{d[e], ix[e]}; }
  __device__ __forceinline__ void set(uint32_t e, const Pair<false>& p) {
    d[e] = p.d;
    ix[e] = p.i;
  }
  __device__ __forceinline__ unsigned long long dist(uint32_t e) const { return d[e]; }
};

// Candidate collection for 32 < k <= CGA_KNN_MAX_K: the warp's buffer of
// `cap` (a power of two, at least 2k) entries in shared memory.  Candidates
// are appended unsorted; whenever the next step could overflow it, or when it
// first holds k, the k-th least distance B is found by bisection on the count
// of entries at most a trial value, every entry beyond B is dropped, and B
// becomes the bound (if ties at B leave too little room, the buffer is
// sorted by a bitonic network and cut to exactly k instead).  Every voxel
// pruned by a bound is beaten by k collected ones, so the final sort's first
// k are the answer.
template <bool NARROW>
struct SmemList {
  using P = Pair<NARROW>;
  using D = typename P::D;
  PairBuf<NARROW> buf;
  uint32_t n, k, cap;

  __device__ __forceinline__ void sort_cut(uint32_t lane) {
    uint32_t S = 32;
    while (S < n) S <<= 1;
    for (uint32_t e = n + lane; e < S; e += 32) buf.set(e, P::none());
    __syncwarp();
    for (uint32_t w = 2; w <= S; w <<= 1) {
      for (uint32_t jj = w >> 1; jj > 0; jj >>= 1) {
        for (uint32_t tt = lane; tt < S / 2; tt += 32) {
          const uint32_t i = ((tt & ~(jj - 1)) << 1) | (tt & (jj - 1)), l = i + jj;
          const P a = buf.get(i), b = buf.get(l);
          const bool up = (i & w) == 0;
          if (up ? b.less(a) : a.less(b)) {
            buf.set(i, b);
            buf.set(l, a);
          }
        }
        __syncwarp();
      }
    }
    n = min(n, k);
  }
  // Keep the entries of distance at most B, the k-th least; returns B.
  __device__ __forceinline__ D select_cut(uint32_t lane) {
    D lo = ~(D)0, hi = 0;
    for (uint32_t e = lane; e < n; e += 32) {
      lo = min(lo, buf.dist(e));
      hi = max(hi, buf.dist(e));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    while (lo < hi) {
      const D mid = lo + ((hi - lo) >> 1);
      uint32_t c = 0;
      for (uint32_t e = lane; e < n; e += 32) c += buf.dist(e) <= mid ? 1u : 0u;
      if (__reduce_add_sync(0xffffffffu, c) >= k) hi = mid; else lo = mid + 1;
    }
    uint32_t out = 0;
    for (uint32_t base = 0; base < n; base += 32) {
      const uint32_t e = base + lane;
      const bool keep = e < n && buf.dist(e) <= lo;
      const P p = keep ? buf.get(e) : P::none();
      const uint32_t bal = __ballot_sync(0xffffffffu, keep);
      __syncwarp();
      if (keep) buf.set(out + __popc(bal & ((1u << lane) - 1u)), p);
      out += __popc(bal);
      __syncwarp();
    }
    n = out;
    if (n + 32 > cap) sort_cut(lane);  // too many ties at B: cut to exactly k
    return lo;
  }
  __device__ __forceinline__ void init(uint32_t kk, uint32_t cp, unsigned char* base, uint32_t wb,
                                       uint32_t warps) {
    buf.init(base, wb, warps, cp);
    n = 0;
    k = kk;
    cap = cp;
  }
  __device__ __forceinline__ D offer(bool has, D cd, uint32_t ci, uint32_t lane, D bound) {
    const uint32_t pending = __ballot_sync(0xffffffffu, has);
    if (has) buf.set(n + __popc(pending & ((1u << lane) - 1u)), P::of(cd, ci));
    n += __popc(pending);
    __syncwarp();
    if (n + 32 > cap || (bound == P::kFar && n >= k)) return select_cut(lane);
    return bound;
  }
  __device__ __forceinline__ void finish(uint32_t lane, size_t row, uint32_t* out_idx,
                                         unsigned long long* out_d2) {
    sort_cut(lane);
    for (uint32_t e = lane; e < k; e += 32) {
      (e < n ? buf.get(e) : P::none()).write(out_idx, out_d2, row + e);
    }
    __syncwarp();
  }
};

// k nearest of one query, one warp: slab rounds as in the NN search (16 per
// side), every lane walking its slab's columns nearest-first in y and each
// column's voxels nearest-first in z.  The lanes step in lockstep, each step
// offering at most one candidate per lane, so that the candidates enter the
// list together and the k-th distance prunes every walk; a lane whose column
// runs out moves to its next column (and offers that column's nearest voxel)
// in the same step.  The narrow form gives up (true) while its list still has room and a
// quarter of the lanes have met what lies beyond its range: without a bound it would go
// through every column within that range, probably for nothing (10k queries up to 65k
// voxels outside a world of 30k surface voxels, b = 16, k = 8: 44.7 ms that way, 4.9 in 64
// bits alone, 7.2 so).
template <bool NARROW, typename L>
__device__ __forceinline__ bool knn_walk(const SearchSeg& sg, const RQuery& q, uint32_t h,
                                         uint32_t lane, L& list) {
  using P = Pair<NARROW>;
  using D = typename P::D;
  const Levels& a = sg.a;
  const int top = (1 << a.bits) - 1;
  const int qx = q.x, qy = q.y, qz = q.z;
  const uint32_t cqy = (uint32_t)min(max(qy, 0), top);
  const uint32_t cqz = (uint32_t)min(max(qz, 0), top);
  const uint32_t cqx = (uint32_t)min(max(qx, 0), top);
  const uint32_t xr0 =
      sg.xdir != nullptr ? __ldg(sg.xdir + cqx) : lower_bound_u16(a.idx2, 0, h, cqx);
  const bool right = (lane & 1u) == 0u;
  D bound = P::kFar;
  for (uint32_t r = 0;; ++r) {
    const int kk = (int)(r * 16u + (lane >> 1));
    const int slab = right ? (int)xr0 + kk : (int)xr0 - 1 - kk;
    bool work = slab >= 0 && slab < (int)h;
    D dx2 = 0;
    uint32_t ys = 0, ye = 0;
    if (work) {
      dx2 = P::square(absdiff32(__ldg(a.idx2 + slab), qx));
      ys = __ldg(a.ptr2 + slab);
      ye = __ldg(a.ptr2 + slab + 1);
      work = dx2 <= bound;
    }
    if (!__any_sync(0xffffffffu, work)) break;
    // column cursors outward from the query's y: [cr, ye) to the right,
    // [ys, cl) to the left; z cursors likewise within the column
    uint32_t cr = 0, cl = 0;
    if (work) {
      cr = lower_bound_u16(a.idx1, ys, ye, cqy);
      cl = cr;
    }
    bool in_col = false;
    D dxy = 0;
    uint32_t zs = 0, ze = 0, zu = 0, zd = 0;
    while (__any_sync(0xffffffffu, work)) {
      bool has = false;
      D cd = P::kFar;
      uint32_t ci = 0xffffffffu;
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        if (work && !has && !in_col) {
          // the next column, nearest in y first, while it can still beat the bound
          const bool hr = cr < ye, hl = cl > ys;
          const uint32_t er = hr ? absdiff32(__ldg(a.idx1 + cr), qy) : 0xffffffffu;
          const uint32_t el = hl ? absdiff32(__ldg(a.idx1 + cl - 1), qy) : 0xffffffffu;
          const bool gr = hr && (!hl || er <= el);
          const D d = P::plus(dx2, P::square(gr ? er : el));
          if ((!hr && !hl) || d > bound) {
            work = false;
          } else {
            const uint32_t c = gr ? cr++ : --cl;
            dxy = d;
            uint32_t clo, chi;
            column_of(a, sg.ctab, c, zs, ze, clo, chi);
            zu = cqz <= clo ? zs : (cqz > chi ? ze : lower_bound_u16(a.idx0, zs, ze, cqz));
            zd = zu;
            in_col = true;
          }
        }
        if (work && !has && in_col) {
          // the column's next voxel, nearest in z first
          const bool hu = zu < ze, hd = zd > zs;
          const uint32_t eu = hu ? absdiff32(__ldg(a.idx0 + zu), qz) : 0xffffffffu;
          const uint32_t ed = hd ? absdiff32(__ldg(a.idx0 + zd - 1), qz) : 0xffffffffu;
          const bool gu = hu && (!hd || eu <= ed);
          const D d = P::plus(dxy, P::square(gu ? eu : ed));
          if ((!hu && !hd) || d > bound) {
            in_col = false;
          } else {
            ci = gu ? zu++ : --zd;
            cd = d;
            has = true;
          }
        }
      }
      bound = list.offer(has, cd, ci, lane, bound);
      if (NARROW && bound == P::kFar) {
        // dropped with columns left, or out of a column with voxels left
        const bool far = work ? !in_col && (zu < ze || zd > zs) : cr < ye || cl > ys;
        if (__popc(__ballot_sync(0xffffffffu, far)) >= 8) return true;
      }
    }
  }
  return false;
}

// The narrow form answers every query; the wide form (a launch after it) the
// queries that the narrow one left with fewer than min(k, u) neighbours, or, on its own,
// all of them (alone).  chunk: queries that a warp of the wide form looks at together.
template <bool LARGE, bool NARROW>
__global__ void __launch_bounds__(LARGE ? kKnnLargeThreads : 256, LARGE ? 1 : CGA_KNN_BLOCKS)
    k_knn(SearchSeg sg, uint32_t k, uint32_t cap, const unsigned long long* __restrict__ order,
          uint32_t* out_idx, unsigned long long* out_d2, uint32_t chunk, bool alone) {
  extern __shared__ __align__(16) unsigned char s_knn[];
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t u = (uint32_t)sg.a.hdr->cnt[0], h = (uint32_t)sg.a.hdr->cnt[2];
  typename std::conditional<LARGE, SmemList<NARROW>, RegList<NARROW>>::type list;
  auto init = [&]() {
    if constexpr (LARGE) {
      list.init(k, cap, s_knn, threadIdx.x >> 5, blockDim.x >> 5);
    } else {
      list.init(k);
    }
  };
  auto answer = [&](uint32_t j) {
    init();
    const RQuery q = radius_query(sg, j);
    if (q.valid && u > 0 && knn_walk<NARROW>(sg, q, h, lane, list)) init();
    list.finish(lane, (size_t)j * k, out_idx, out_d2);
  };
  if constexpr (NARROW) {
    constexpr uint32_t W = (LARGE ? kKnnLargeThreads : 256) / 32;
    __shared__ uint32_t s_next;
    open_slots<W>(&s_next);
    for (uint32_t turn = threadIdx.x >> 5;; turn = next_turn(&s_next)) {
      const uint32_t sl = slot_of_turn<W>(turn);
      if (sl >= sg.m) break;
      answer(slot_query(order, sl));
    }
  } else {
    const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    const uint32_t need = min(k, u);
    if (need == 0 && !alone) return;
    for (uint32_t s0 = w * chunk; s0 < sg.m; s0 += nw * chunk) {
      const bool in = lane < chunk && s0 + lane < sg.m;
      const uint32_t j = in ? slot_query(order, s0 + lane) : 0u;
      const bool open = in && (alone || (out_idx[(size_t)j * k + need - 1] == 0xffffffffu &&
                                         radius_query(sg, j).valid));
      uint32_t todo = __ballot_sync(0xffffffffu, open);
      while (todo) {
        answer(__shfl_sync(0xffffffffu, j, __ffs(todo) - 1));
        todo &= todo - 1;
      }
    }
  }
}

// Blocks for m queries.  Up to four waves of them each warp takes one query; beyond,
// four waves or 16 queries a warp on average, whichever are more blocks: within a block
// the warps even their queries out (slot_of_turn), and blocks start where others end, so
// that slow queries, which lie side by side in the order, do not all start late in the
// same blocks.  8 nearest in LiDAR worlds, ms, in one wave and so: 100k queries of 1.3M
// points, b = 16, 1.40 and 0.94 (one warp a query 1.32, 4 queries a warp 1.28), 1M 5.57 and
// 5.52; 10k far from 300k points, b = 13, 18.2 and 12.9; the radius search is the same.
unsigned search_blocks(uint64_t m, unsigned per_sm) {
  const uint64_t all = (std::max<uint64_t>(m, 1) + 7) / 8, wave = (uint64_t)device_sm_count() * per_sm;
  return (unsigned)std::min<uint64_t>(all, std::max<uint64_t>(4 * wave, all / 16));
}

}  // namespace

// Buffer entries per warp for k > 32: the least power of two >= 2k.
static uint32_t knn_cap(uint32_t k) {
  uint32_t c = 64;
  while (c < 2 * k) c <<= 1;
  return c;
}

template <bool NARROW>
static cudaError_t knn_large_attr() {
  return cudaFuncSetAttribute(k_knn<true, NARROW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)((kKnnLargeThreads / 32) * knn_cap(kKnnMaxK) *
                                    PairBuf<NARROW>::kBytes));
}

// The wide form alone answers calls of few queries (each has a warp of its own) whose
// walks are short, of few neighbours or in few voxels: there the second launch costs more
// than 32-bit arithmetic saves.  So it does of few queries on 16-bit grids, where all of
// them may have to be answered twice (100 far from 300k surface voxels, k = 8: 34.6 ms by
// both forms, 17.1 by the wide one).  us by both forms and by the wide one: a query of 50
// voxels, k = 1 29 and 25, k = 16 31 and 27; of 300k LiDAR voxels, b = 13, k = 16 34 and 37;
// 100 queries of those, k = 1 32.5 and 31.5, k = 16 42 and 45.
constexpr uint32_t kKnnAlone = 512, kKnnAloneK = 4, kKnnAloneVoxels = 4096;

cudaError_t run_knn(const SearchSeg& sg, uint32_t k, const unsigned long long* order, uint32_t* idx,
                    unsigned long long* d2, cudaStream_t stream) {
  if (sg.m == 0) return cudaSuccess;
  const uint32_t sms = (uint32_t)device_sm_count();
  const bool alone = sg.m <= kKnnAlone && (k <= kKnnAloneK || sg.a.cap <= kKnnAloneVoxels ||
                                            sg.a.bits == 16);
  // the wide form's check reads one word a query; as many warps as there are share them
  auto chunk = [&](uint64_t warps) {
    return (uint32_t)std::min<uint64_t>((sg.m + warps - 1) / warps, 32);
  };
  if (k <= 32) {
    const unsigned blocks = search_blocks(sg.m, CGA_KNN_BLOCKS);
    if (!alone) k_knn<false, true><<<blocks, 256, 0, stream>>>(sg, k, 0, order, idx, d2, 0, false);
    k_knn<false, false><<<blocks, 256, 0, stream>>>(sg, k, 0, order, idx, d2,
                                                    chunk((uint64_t)blocks * 8), alone);
  } else {
    const uint32_t cap = knn_cap(k), warps = kKnnLargeThreads / 32;
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
      attr = knn_large_attr<true>();
      if (attr == cudaSuccess) attr = knn_large_attr<false>();
    });
    if (attr != cudaSuccess) return attr;
    // one wave: what shared memory (and 64 registers a thread) lets an SM hold
    auto blocks = [&](size_t smem) {
      const uint32_t per_sm =
          std::max<uint32_t>(1, std::min<uint32_t>(8, (uint32_t)((220u << 10) / (smem + 1024))));
      return (unsigned)std::min<uint64_t>((sg.m + warps - 1) / warps, sms * per_sm);
    };
    const size_t smem = (size_t)warps * cap * PairBuf<true>::kBytes;
    const size_t wide = (size_t)warps * cap * PairBuf<false>::kBytes;
    if (!alone) {
      k_knn<true, true><<<blocks(smem), kKnnLargeThreads, smem, stream>>>(sg, k, cap, order, idx, d2,
                                                                         0, false);
    }
    k_knn<true, false><<<blocks(wide), kKnnLargeThreads, wide, stream>>>(
        sg, k, cap, order, idx, d2, chunk((uint64_t)blocks(wide) * warps), alone);
  }
  count_launch(alone ? 1 : 2);
  return cudaGetLastError();
}

// Radii whose squared distances fit 32 bits.
constexpr unsigned long long kNarrowRadius2 = 1ull << 31;

// Largest s with s * s <= v (v <= 2^62).
static unsigned long long host_isqrt(unsigned long long v) {
  unsigned long long s = (unsigned long long)std::sqrt((double)v);
  while (s > 0 && s * s > v) --s;
  while ((s + 1) * (s + 1) <= v) ++s;
  return s;
}

size_t radius_scratch_bytes() { return 1025 * sizeof(unsigned long long); }

cudaError_t run_radius_count(const SearchSeg& sg, unsigned long long r2,
                             const unsigned long long* order, unsigned long long* offsets,
                             void* scratch, cudaStream_t stream) {
  unsigned long long* totals = static_cast<unsigned long long*>(scratch);
  if (sg.m > 0) {
    if (r2 < kNarrowRadius2) {
      k_radius_count<uint32_t><<<search_blocks(sg.m, CGA_RADIUS_BLOCKS), 256, 0, stream>>>(
          sg, (uint32_t)r2, (uint32_t)host_isqrt(r2), order, offsets);
    } else {
      k_radius_count<unsigned long long><<<search_blocks(sg.m, CGA_RADIUS_BLOCKS), 256, 0, stream>>>(
          sg, r2, host_isqrt(r2), order, offsets);
    }
  }
  const uint32_t B = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(1024, (sg.m + 4095) / 4096));
  const uint64_t chunk = (sg.m + B - 1) / B;
  k_scan_totals<<<B, kThreads, 0, stream>>>(offsets, sg.m, std::max<uint64_t>(chunk, 1), totals);
  k_scan_top<<<1, kThreads, 0, stream>>>(totals, B);
  k_scan_apply<<<B, kThreads, 0, stream>>>(offsets, sg.m, std::max<uint64_t>(chunk, 1), totals, B);
  count_launch(sg.m > 0 ? 4 : 3);
  return cudaGetLastError();
}

cudaError_t run_radius_fill(const SearchSeg& sg, unsigned long long r2,
                            const unsigned long long* order, const unsigned long long* offsets,
                            uint32_t* idx, unsigned long long* d2, cudaStream_t stream) {
  if (sg.m == 0) return cudaSuccess;
  if (r2 < kNarrowRadius2) {
    k_radius_fill<uint32_t><<<search_blocks(sg.m, CGA_RADIUS_BLOCKS), 256, 0, stream>>>(
        sg, (uint32_t)r2, (uint32_t)host_isqrt(r2), order, offsets, idx, d2);
  } else {
    k_radius_fill<unsigned long long><<<search_blocks(sg.m, CGA_RADIUS_BLOCKS), 256, 0, stream>>>(
        sg, r2, host_isqrt(r2), order, offsets, idx, d2);
  }
  count_launch(1);
  return cudaGetLastError();
}

}  // namespace libcga
