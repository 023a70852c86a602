// Sort pipeline of the CGA build (and of the xz / yz projections): builds from points
// go by bins where plan_bins says so (k_bins.cuh), the others, and what the bins leave
// over (k_lsd_all, all of the following in one launch), by LSD radix passes:
//   k_seg_init     headers and empty-CGA sentinels
//   k_keys_hist    quantize (+ rigid transform) and encode each point, or (k_keys_walk)
//                  re-key a CGA point for a projection; per-segment digit
//                  histograms of every radix pass in the same read
//   k_onesweep     one LSD radix pass: warp-level digit ranking, decoupled
//                  look-back over tiles for the global digit offsets, scatter
//   k_compact      dedupe + CGA compaction (k_compact.cuh)
// Every kernel works on a batch of segments (clouds); a tile never spans two
// segments and look-back chains stop at the segment's first tile.
#include <algorithm>
#include <mutex>

#include "k_bins.cuh"
#include "k_compact.cuh"
#include "k_walk.cuh"

namespace libcga {

namespace {

// Element count of a segment: known on the host for a build, read from the
// source header for a projection (the source is built earlier in the stream).
__device__ __forceinline__ uint32_t seg_count(const SortSeg& s) {
  if (s.from_cga) return (uint32_t)s.src.hdr->cnt[0];
  return s.n_host;
}

__global__ void k_seg_init(const SortSeg* __restrict__ segs, int S) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  const Levels& o = segs[s].out;
  o.hdr->cnt[0] = 0;
  o.hdr->cnt[1] = 0;
  o.hdr->cnt[2] = 0;
  o.hdr->err = segs[s].from_cga ? segs[s].src.hdr->err : 0u;
  o.ptr1[0] = 0;
  if (o.nlevels == 3) o.ptr2[0] = 0;
}

// The digit counts of a block's current segment, in shared memory, and their way to the
// segment's histogram (digits of RB bits).
template <int RB>
struct BlockHist {
  uint32_t cnt[kMaxPasses][1 << RB];
  uint32_t err;

  __device__ __forceinline__ void open() {
    for (int i = threadIdx.x; i < kMaxPasses << RB; i += kThreads) (&cnt[0][0])[i] = 0;
    if (threadIdx.x == 0) err = 0;
    __syncthreads();
  }
  __device__ __forceinline__ void flush(const SortSeg* __restrict__ segs, int s, uint32_t* hist) {
    __syncthreads();
    const uint32_t passes = segs[s].passes;
    for (int i = threadIdx.x; i < kMaxPasses << RB; i += kThreads) {
      const uint32_t v = (&cnt[0][0])[i];
      if (v != 0 && (uint32_t)(i >> RB) < passes) {
        atomicAdd(hist + ((size_t)s * kMaxPasses << RB) + i, v);
      }
      (&cnt[0][0])[i] = 0;
    }
    if (threadIdx.x == 0 && err) {
      atomicOr(&segs[s].out.hdr->err, err);
      err = 0;
    }
    __syncthreads();
  }
};

// Keys of the points of the tiles [t0, t1) plus per-segment histograms of every pass.
// marked: only the segments marked for the general sort.
template <typename K, int RB>
__device__ __forceinline__ void keys_hist_tiles(const SortSeg* __restrict__ segs, int S,
                                                uint32_t t0, uint32_t t1, K* keys0,
                                                uint32_t* hist, bool marked) {
  __shared__ BlockHist<RB> sh;
  __shared__ float s_pts[kThreads * 3];
  const int tid = threadIdx.x;
  if (t0 >= t1) return;
  sh.open();
  int cur = find_seg(segs, S, t0);
  for (uint32_t t = t0; t < t1; ++t) {
    const int s = find_seg(segs, S, t);
    if (s != cur) {
      sh.flush(segs, cur, hist);
      cur = s;
    }
    const SortSeg& sg = segs[s];
    if (marked && !sg.fallback) continue;
    const uint32_t n = sg.n_host;
    const uint32_t start = (t - sg.tile_base) * kTile;
    if (start >= n) continue;
    const uint32_t cnt = min((uint32_t)kTile, n - start);
    K* out = keys0 + sg.key_base + start;
    const uint32_t passes = sg.passes;
    const float* src = sg.xyz + (size_t)start * 3;
    for (uint32_t c0 = 0; c0 < cnt; c0 += kThreads) {
      const uint32_t m = min((uint32_t)kThreads, cnt - c0);
      __syncthreads();
      for (uint32_t i = tid; i < m * 3; i += kThreads) s_pts[i] = __ldg(src + (size_t)c0 * 3 + i);
      __syncthreads();
      if ((uint32_t)tid < m) {
        K key;
        if (!point_key<K>(s_pts[3 * tid], s_pts[3 * tid + 1], s_pts[3 * tid + 2],
                          sg.has_x != 0, sg.X, sg.scale, sg.off, sg.bits, key)) {
          atomicOr(&sh.err, kErrNonfinite);
        }
        out[c0 + tid] = key;
        for (uint32_t p = 0; p < passes; ++p) {
          atomicAdd(&sh.cnt[p][(uint32_t)(key >> (sg.bit0 + p * RB)) & ((1 << RB) - 1)], 1u);
        }
      }
    }
  }
  sh.flush(segs, cur, hist);
}

template <typename K, int RB>
__global__ void __launch_bounds__(kThreads) k_keys_hist(const SortSeg* __restrict__ segs, int S,
                                                        uint32_t total_tiles,
                                                        uint32_t tiles_per_cta, K* keys0,
                                                        uint32_t* hist) {
  const uint32_t t0 = blockIdx.x * tiles_per_cta;
  keys_hist_tiles<K, RB>(segs, S, t0, min(t0 + tiles_per_cta, total_tiles), keys0, hist, false);
}

// The same for segments whose keys come from a CGA (projections, coarse levels, trees): a
// block takes runs of a step of a walk for each of its warps (k_walk.cuh), not whole tiles,
// so that small sources have a warp for every step: the xz projection of 30k points at b =
// 16 took 96 us by tiles, 79 so.  Eight blocks an SM hide more of the walk's loads than
// four (the tree of 20M surface voxels 1595 us, five 1562, six 1575, eight 1540).
constexpr int kKeysWalkPerSm = 8;
constexpr uint32_t kWalkRun = kWarps * kWalk;
static_assert(kTile % kWalkRun == 0, "runs of a tile");
template <typename K, int RB>
__global__ void __launch_bounds__(kThreads, kKeysWalkPerSm)
    k_keys_walk(const SortSeg* __restrict__ segs, int S, uint32_t total_runs, uint32_t runs_per_cta,
                K* keys0, uint32_t* hist) {
  constexpr uint32_t PER = kTile / kWalkRun;
  __shared__ BlockHist<RB> sh;
  const uint32_t r1 = min((blockIdx.x + 1) * runs_per_cta, total_runs);
  uint32_t r = blockIdx.x * runs_per_cta;
  if (r >= r1) return;
  sh.open();
  while (r < r1) {
    // the block's runs of one segment, a warp per equal share of their positions
    const int s = find_seg(segs, S, r / PER);
    const SortSeg& sg = segs[s];
    const Levels& a = sg.src;
    const uint32_t n = (uint32_t)a.hdr->cnt[0], b = sg.bits, passes = sg.passes;
    const uint32_t base = sg.tile_base * PER, re = min(r1, base + sg.num_tiles * PER);
    const uint32_t start = min(n, (r - base) * kWalkRun), stop = min(n, (re - base) * kWalkRun);
    const uint32_t per = ((stop - start + kWalkRun - 1) / kWalkRun) * kWalk;
    const uint32_t w0 = min(stop, start + (threadIdx.x >> 5) * per);
    K* kout = keys0 + sg.key_base;
    walk_voxels(a, w0, min(stop, w0 + per), [&](uint32_t p, uint32_t valid, const uint32_t* x,
                                                const uint32_t* y, const uint32_t* z) {
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) {
        K key;
        if (sg.plane == 3) {
          const uint32_t L = sg.shift;
          key = ((K)(x[i] >> L) << (2 * b)) | ((K)(y[i] >> L) << b) | (K)(z[i] >> L);
        } else if (sg.plane == 4) {
          key = (K)tree_key(x[i], y[i], z[i], sg.shift);
        } else {
          const uint32_t u = sg.plane == 2 ? y[i] : x[i], v = sg.plane == 0 ? y[i] : z[i];
          key = ((K)u << b) | (K)v;
        }
        const bool ok = (valid >> i) & 1u;
        if (ok) kout[p + 32 * i + (threadIdx.x & 31)] = key;
        // neighbouring voxels share their high digits: one count for the
        // warp where all lanes hold the same digit
        const uint32_t live = __ballot_sync(0xffffffffu, ok);
        for (uint32_t q = 0; q < passes; ++q) {
          const uint32_t d = (uint32_t)(key >> (sg.bit0 + q * RB)) & ((1 << RB) - 1);
          const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
          if (__all_sync(0xffffffffu, !ok || d == d0)) {
            if ((threadIdx.x & 31) == 0 && live) atomicAdd(&sh.cnt[q][d0], (uint32_t)__popc(live));
          } else if (ok) {
            atomicAdd(&sh.cnt[q][d], 1u);
          }
        }
      }
    });
    sh.flush(segs, s, hist);
    r = re;
  }
}

// Dynamic shared memory of one pass block: the tile's keys, per-warp digit
// counts (u16), per-digit offsets and the warp scan words.
template <typename K, int TH, int RB>
constexpr size_t onesweep_smem() {
  return (size_t)kTile * sizeof(K) + (size_t)(TH / 32) * (1 << RB) * 2 + (size_t)(1 << RB) * 4 +
         (size_t)(TH / 32) * 4;
}

// Blocks per SM a pass kernel is compiled for (its register budget), per
// threads per tile; measured on GB300 (30M-key builds): more resident warps
// hide more of the key loads and look-back waits than the few spilled values
// cost.
#ifndef CGA_SORT_BLOCKS_512
#define CGA_SORT_BLOCKS_512 4
#endif
#ifndef CGA_SORT_BLOCKS_256
#define CGA_SORT_BLOCKS_256 5
#endif

// One tile of an LSD pass over digit `pass` (RB bits): kTile keys as TH threads
// x kTile/TH keys (warp-striped); threads tid < 2^RB own one digit each for the
// per-digit steps.
template <typename K, int TH, int RB>
__device__ __forceinline__ void onesweep_tile(const SortSeg* __restrict__ segs, int s, uint32_t t,
                                              int pass, const K* __restrict__ in,
                                              K* __restrict__ out,
                                              const uint32_t* __restrict__ hist, uint32_t* look) {
  constexpr int IT = kTile / TH, WARPS = TH / 32, R = 1 << RB;
  static_assert(IT * TH == kTile && TH >= R, "tile shape");
  extern __shared__ __align__(16) unsigned char s_raw[];
  K* s_keys = reinterpret_cast<K*>(s_raw);
  uint16_t (*s_wh)[R] = reinterpret_cast<uint16_t (*)[R]>(s_raw + (size_t)kTile * sizeof(K));
  uint32_t* s_off = reinterpret_cast<uint32_t*>(s_raw + (size_t)kTile * sizeof(K) +
                                                (size_t)WARPS * R * 2);
  uint32_t* s_scan = s_off + R;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int i = tid; i < WARPS * R; i += TH) (&s_wh[0][0])[i] = 0;
  __syncthreads();
  const SortSeg& sg = segs[s];
  if (pass >= (int)sg.passes) return;
  const uint32_t n = seg_count(sg);
  const uint32_t lt = t - sg.tile_base;
  const uint32_t start = lt * kTile;
  if (start >= n) return;
  const uint32_t cnt = min((uint32_t)kTile, n - start);
  const K* src = in + sg.key_base + start;
  const int shift = (int)sg.bit0 + pass * RB;

  K k[IT];
  uint32_t dg[IT], rk[IT];
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    const uint32_t e = (uint32_t)(w * 32 * IT + i * 32 + lane);
    const bool v = e < cnt;
    k[i] = v ? src[e] : (K)0;
    dg[i] = v ? ((uint32_t)(k[i] >> shift) & (R - 1)) : 0xffffffffu;
  }
  // warp-level ranking: lanes holding the same digit form one peer group
  uint16_t* wh = s_wh[w];
  const uint32_t ltm = lanemask_lt();
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    const uint32_t d = dg[i];
    // lanes with the same digit: one warp vote per digit bit and one for
    // validity (votes issue faster than a match over the digit)
    uint32_t peers = __ballot_sync(0xffffffffu, d < (uint32_t)R);
    if (d >= (uint32_t)R) peers = ~peers;
#pragma unroll
    for (int bit = 0; bit < RB; ++bit) {
      const uint32_t v = __ballot_sync(0xffffffffu, (d >> bit) & 1u);
      peers &= ((d >> bit) & 1u) ? v : ~v;
    }
    const uint32_t base = (d < (uint32_t)R) ? wh[d] : 0u;
    __syncwarp();
    if (d < (uint32_t)R && lane == __ffs(peers) - 1) wh[d] = (uint16_t)(base + __popc(peers));
    __syncwarp();
    rk[i] = base + __popc(peers & ltm);
  }
  __syncthreads();
  // per digit (thread tid == digit): warp offsets, tile count, publish
  const int d = tid;
  const bool owner = tid < R;
  uint32_t tile_cnt = 0;
  uint32_t* my = look + (size_t)t * R + d;
  if (owner) {
    for (int x = 0; x < WARPS; ++x) {
      const uint32_t v = s_wh[x][d];
      s_wh[x][d] = (uint16_t)tile_cnt;
      tile_cnt += v;
    }
    st_relaxed(my, (lt == 0 ? kFlagInc : kFlagAgg) | tile_cnt);
  }
  uint32_t tot;
  const uint32_t bin_start = block_scan_th<TH>(owner ? tile_cnt : 0u, tot, s_scan);
  const uint32_t hv = owner ? hist[((size_t)s * kMaxPasses + pass) * R + d] : 0u;
  const uint32_t dbase = block_scan_th<TH>(hv, tot, s_scan);
  if (owner) s_off[d] = bin_start;
  __syncthreads();
  bool bad = false;
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    if (dg[i] < (uint32_t)R) {
      const uint32_t pos = s_off[dg[i]] + s_wh[w][dg[i]] + rk[i];
      if (pos < (uint32_t)kTile) s_keys[pos] = k[i]; else bad = true;
    }
  }
  uint32_t excl = 0;
  if (owner && lt > 0) {
    excl = lookback(look + d, R, t, sg.tile_base, &sg.out.hdr->err);
    st_relaxed(my, kFlagInc | ((excl + tile_cnt) & kValMask));
  }
  __syncthreads();
  if (owner) s_off[d] = dbase + excl - bin_start;
  __syncthreads();
  K* dst = out + sg.key_base;
  for (uint32_t e = tid; e < cnt; e += TH) {
    const K key = s_keys[e];
    const uint32_t pos = s_off[(uint32_t)(key >> shift) & (R - 1)] + e;
    if (pos < n) dst[pos] = key; else bad = true;
  }
  if (bad) atomicOr(&sg.out.hdr->err, kErrInternal);
}

// One LSD pass over every segment that still needs it, a tile per block.
template <typename K, int TH, int RB>
__global__ void __launch_bounds__(TH, TH == 512 ? CGA_SORT_BLOCKS_512 : CGA_SORT_BLOCKS_256)
    k_onesweep(const SortSeg* __restrict__ segs, int S, int pass, const K* __restrict__ in,
               K* __restrict__ out, const uint32_t* __restrict__ hist, uint32_t* look,
               uint32_t* counter) {
  __shared__ uint32_t s_tile;
  __shared__ int s_seg;
  if (threadIdx.x == 0) {
    const uint32_t t = atomicAdd(counter, 1u);
    s_tile = t;
    s_seg = find_seg(segs, S, t);
  }
  __syncthreads();
  onesweep_tile<K, TH, RB>(segs, s_seg, s_tile, pass, in, out, hist, look);
}

// Dedupe and compaction of one tile of sorted keys (src: the segment's sorted
// key buffer).
template <typename K, int LEVELS>
__device__ __forceinline__ void compact_sorted_tile(const SortSeg& sg, uint32_t t,
                                                    const K* __restrict__ sorted,
                                                    uint32_t* clook, CompactSmem& sm) {
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const uint32_t n = seg_count(sg);
  const uint32_t lt = t - sg.tile_base;
  const uint32_t start = lt * kTile;
  if (start >= n) return;
  const uint32_t cnt = min((uint32_t)kTile, n - start);
  const K* src = sorted + sg.key_base + start;
  K k[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t e = (uint32_t)(w * 32 * kItems + i * 32 + lane);
    k[i] = (e < cnt) ? src[e] : (K)0;
  }
  const bool has_prev = start > 0;
  const K prev = has_prev ? src[-1] : (K)0;
  const bool last = (start + cnt == n);
  compact_tile<LEVELS, K>(k, cnt, has_prev, prev, t, sg.tile_base, last, sg.out, clook, sm);
}

template <typename K, int LEVELS>
__global__ void __launch_bounds__(kThreads) k_compact(const SortSeg* __restrict__ segs, int S,
                                                      const K* __restrict__ keys0,
                                                      const K* __restrict__ keys1,
                                                      uint32_t* clook, uint32_t* counter) {
  __shared__ CompactSmem sm;
  __shared__ uint32_t s_tile;
  __shared__ int s_seg;
  if (threadIdx.x == 0) {
    const uint32_t t = atomicAdd(counter, 1u);
    s_tile = t;
    s_seg = find_seg(segs, S, t);
  }
  __syncthreads();
  const SortSeg& sg = segs[s_seg];
  compact_sorted_tile<K, LEVELS>(sg, s_tile, (sg.passes & 1u) ? keys1 : keys0, clook, sm);
}

// The general sort of the segments that a build by bins marked (usually none: the
// blocks look and leave): clearing of the tables, key generation, the 8-bit radix passes
// and the compaction in one launch, as phases of items (wait_done).  The tables of the
// bins lie in the look-back words, so those are cleared here.
constexpr int kLsdTurn = kMaxPasses + 2, kLsdDone = kMaxPasses + 4;  // words of the counters
static_assert(kLsdDone < kCounterWords, "counters");
constexpr uint32_t kLsdZero = 16384;  // words cleared by an item
template <typename K>
__global__ void __launch_bounds__(kThreads, 4)
    k_lsd_all(SortSeg* segs, int S, uint32_t total_tiles, uint32_t max_passes, K* keys0, K* keys1,
              uint32_t* hist, uint32_t* look, uint32_t* clook, uint32_t* counters,
              uint32_t zero_words) {
  __shared__ CompactSmem sm;
  __shared__ uint32_t s_item;
  __shared__ int s_seg;
  const uint32_t tid = threadIdx.x;
  int any = 0;
  for (int s = (int)tid; s < S; s += kThreads) any |= (int)segs[s].fallback;
  if (!__syncthreads_or(any)) return;
  unsigned int* err = &segs[0].out.hdr->err;
  // items: hist, look and clook, which lie side by side, in runs of words; keys, a share of
  // the tiles each; a tile each for every pass and for the compaction
  const uint32_t nz = (zero_words + kLsdZero - 1) / kLsdZero;
  const uint32_t nk = min(gridDim.x, total_tiles), per = (total_tiles + nk - 1) / nk;
  uint32_t open = 0;  // the last phase known to have begun
  for (;;) {
    __syncthreads();  // the previous item's shared data is read no more
    if (tid == 0) s_item = atomicAdd(counters + kLsdTurn, 1u);
    __syncthreads();
    uint32_t i = s_item, before = 0, phase = 0;
    if (i >= nz + nk) {
      const uint32_t q = (i - nz - nk) / total_tiles;
      if (q > max_passes) return;
      phase = 2 + q;
      before = nz + nk + q * total_tiles;
    } else if (i >= nz) {
      phase = 1;
      before = nz;
    }
    i -= before;
    if (phase > open) {
      if (!wait_done(counters + kLsdDone, before, err)) return;
      open = phase;
    }
    if (phase == 0) {
      const uint32_t w1 = min(zero_words, (i + 1) * kLsdZero);
      for (uint32_t w = i * kLsdZero + tid; w < w1; w += kThreads) hist[w] = 0;
    } else if (phase == 1) {
      keys_hist_tiles<K, 8>(segs, S, i * per, min((i + 1) * per, total_tiles), keys0, hist, true);
    } else {
      const uint32_t p = phase - 2;  // pass p, and after the last one the compaction
      if (tid == 0) s_seg = find_seg(segs, S, i);
      __syncthreads();
      const SortSeg& sg = segs[s_seg];
      if (sg.fallback && p < max_passes) {
        onesweep_tile<K, kThreads, 8>(segs, s_seg, i, (int)p, (p & 1) ? keys1 : keys0,
                                      (p & 1) ? keys0 : keys1, hist,
                                      look + ((size_t)p * total_tiles << 8));
      } else if (sg.fallback) {
        compact_sorted_tile<K, 3>(sg, i, (sg.passes & 1u) ? keys1 : keys0, clook, sm);
      }
    }
    count_done(counters + kLsdDone);
  }
}

size_t align_up(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace

size_t sort_scratch_bytes(uint64_t total_keys, uint32_t total_tiles, int S, bool key64,
                          uint32_t radix_bits) {
  const size_t ks = key64 ? 8 : 4;
  const size_t R = (size_t)1 << radix_bits;
  size_t b = 0;
  b += align_up(total_keys * ks) * 2;
  b += align_up((size_t)S * kMaxPasses * R * 4);
  b += align_up((size_t)kMaxPasses * total_tiles * R * 4);
  b += align_up((size_t)total_tiles * 3 * 4);
  b += align_up(kCounterWords * 4);
  b += align_up((size_t)S * sizeof(SortSeg));
  return b;
}

SortScratch sort_scratch_carve(void* base, uint64_t total_keys, uint32_t total_tiles, int S,
                               bool key64, const Tuning& tu) {
  const size_t ks = key64 ? 8 : 4;
  const size_t R = (size_t)1 << tu.radix_bits;
  char* p = static_cast<char*>(base);
  SortScratch sc{};
  sc.radix_bits = tu.radix_bits;
  sc.sort_threads = tu.sort_threads;
  sc.keys0 = p;
  p += align_up(total_keys * ks);
  sc.keys1 = p;
  p += align_up(total_keys * ks);
  char* z0 = p;
  sc.hist = reinterpret_cast<uint32_t*>(p);
  p += align_up((size_t)S * kMaxPasses * R * 4);
  sc.look = reinterpret_cast<uint32_t*>(p);
  p += align_up((size_t)kMaxPasses * total_tiles * R * 4);
  sc.clook = reinterpret_cast<uint32_t*>(p);
  p += align_up((size_t)total_tiles * 3 * 4);
  sc.counters = reinterpret_cast<uint32_t*>(p);
  p += align_up(kCounterWords * 4);
  sc.zero_bytes = (size_t)(p - z0);
  sc.segs = reinterpret_cast<SortSeg*>(p);
  return sc;
}

int device_sm_count() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  return sms;
}

template <typename K, int TH, int RB>
static cudaError_t set_pass_smem() {
  return cudaFuncSetAttribute(k_onesweep<K, TH, RB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)onesweep_smem<K, TH, RB>());
}

template <typename K, int TH, int RB>
static void launch_shape(int S, uint32_t total_tiles, uint32_t max_passes, const SortScratch& sc,
                         cudaStream_t stream) {
  K* k0 = static_cast<K*>(sc.keys0);
  K* k1 = static_cast<K*>(sc.keys1);
  constexpr size_t smem = onesweep_smem<K, TH, RB>();
  for (uint32_t p = 0; p < max_passes; ++p) {
    const K* in = (p & 1) ? k1 : k0;
    K* out = (p & 1) ? k0 : k1;
    k_onesweep<K, TH, RB><<<total_tiles, TH, smem, stream>>>(
        sc.segs, S, (int)p, in, out, sc.hist, sc.look + ((size_t)p * total_tiles << RB),
        sc.counters + p);
  }
  count_launch(max_passes);
}

template <typename K>
static void launch_passes(int S, uint32_t total_tiles, uint32_t max_passes, const SortScratch& sc,
                          cudaStream_t stream) {
  if (sc.radix_bits == 9) {
    launch_shape<K, 512, 9>(S, total_tiles, max_passes, sc, stream);
  } else if (sc.sort_threads == 256) {
    launch_shape<K, 256, 8>(S, total_tiles, max_passes, sc, stream);
  } else {
    launch_shape<K, 512, 8>(S, total_tiles, max_passes, sc, stream);
  }
}

// Resident blocks of the bin kernels (set by init_bin_kernels): the job sorts of
// 32- and 64-bit keys, and the general sort behind them.
static uint32_t g_bin_sort_blocks[2], g_lsd_blocks[2], g_bin_values_blocks[2];

template <typename F>
static cudaError_t resident(F* kernel, int threads, size_t smem, uint32_t* blocks) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int n = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem);
  if (e == cudaSuccess && n <= 0) e = cudaErrorInvalidConfiguration;
  if (blocks != nullptr) *blocks = (uint32_t)std::max(n, 1) * (uint32_t)device_sm_count();
  return e;
}

static cudaError_t init_bin_kernels() {
  const cudaError_t es[] = {
      resident(k_bin_sort<uint32_t>, kBinThreads, bin_sort_smem<uint32_t>(), &g_bin_sort_blocks[0]),
      resident(k_bin_sort<unsigned long long>, kBinThreads, bin_sort_smem<unsigned long long>(),
               &g_bin_sort_blocks[1]),
      resident(k_bin_part<uint32_t, 4, false>, 1024, bin_part_smem<uint32_t, 4>(), nullptr),
      resident(k_bin_part<uint32_t, 4, true>, 1024, bin_part_smem<uint32_t, 4>(), nullptr),
      resident(k_bin_part<uint32_t, 8, false>, 1024, bin_part_smem<uint32_t, 8>(), nullptr),
      resident(k_bin_part<uint32_t, 8, true>, 1024, bin_part_smem<uint32_t, 8>(), nullptr),
      resident(k_bin_part<uint32_t, 16, false>, 1024, bin_part_smem<uint32_t, 16>(), nullptr),
      resident(k_bin_part<uint32_t, 16, true>, 1024, bin_part_smem<uint32_t, 16>(), nullptr),
      resident(k_bin_part<unsigned long long, 4, false>, 1024, bin_part_smem<unsigned long long, 4>(), nullptr),
      resident(k_bin_part<unsigned long long, 4, true>, 1024, bin_part_smem<unsigned long long, 4>(), nullptr),
      resident(k_bin_part<unsigned long long, 8, false>, 1024, bin_part_smem<unsigned long long, 8>(), nullptr),
      resident(k_bin_part<unsigned long long, 8, true>, 1024, bin_part_smem<unsigned long long, 8>(), nullptr),
      resident(k_bin_part<unsigned long long, 16, false>, 1024, bin_part_smem<unsigned long long, 16>(), nullptr),
      resident(k_bin_part<unsigned long long, 16, true>, 1024, bin_part_smem<unsigned long long, 16>(), nullptr),
      resident(k_bin_values<uint32_t>, kBinThreads, bin_values_smem<uint32_t>(),
               &g_bin_values_blocks[0]),
      resident(k_bin_values<unsigned long long>, kBinThreads,
               bin_values_smem<unsigned long long>(), &g_bin_values_blocks[1]),
      resident(k_lsd_all<uint32_t>, kThreads, onesweep_smem<uint32_t, kThreads, 8>(), &g_lsd_blocks[0]),
      resident(k_lsd_all<unsigned long long>, kThreads,
               onesweep_smem<unsigned long long, kThreads, 8>(), &g_lsd_blocks[1])};
  for (cudaError_t e : es) {
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Points per segment up to which a build goes by bins: beyond, a bin of the
// widest table (2^12) holds more than a block sorts.
constexpr uint64_t kBinMaxPoints = 1ull << 25;
// On grids of at most 8 bits (no more than three digits to sort) a bin is a slab or more
// and most clouds leave most of them empty: by bins only up to 512 points a bin, and again,
// at 7 and 8 bits, where all of them have to be split anyway.  By bins and in general, us: 300k LiDAR points, b = 5 132 and 76, b = 8 106 and 89, uniform ones 93
// and 73, 80 and 95; 1M surface points, b = 6 136 and 106, b = 8 115 and 107; 130k LiDAR
// points, b = 7 94 and 80; 30k uniform ones, b = 7, 56 and 67; 3M, b = 8, 186 and 204.  (With attributes by bins all
// the same: their sums cost more in general.  1M LiDAR points, b = 6 357 and 819.)
constexpr uint32_t kBinCoarseBits = 8;
constexpr uint64_t kBinCoarsePoints = 512, kBinCoarseMost = 8192;
static bool coarse_build(const SortSeg& g) {
  return g.bits <= kBinCoarseBits && g.n_host >= kBinCoarsePoints << g.bits &&
         (g.bits <= 6 || g.n_host < kBinCoarseMost << g.bits);
}

void plan_bins(SortSeg* h_segs, int S, uint32_t total_tiles, SortScratch& sc, bool values) {
  BinPlan& B = sc.bins;
  B = BinPlan{};
  if (S <= 0 || total_tiles == 0) return;
  // bins of about 64 points, no finer than a slab (whole slabs per bin), and 32-bit
  // keys where a bin and 32 bits give the key with room for four bins a job.  On
  // average a bin may hold a few blocks' worth of points (30M points at b = 10, 29k a
  // bin: 1377 us by the general sort, 1368 by bins); beyond that every bin goes to a
  // cluster, which the general sort beats (15k a bin that way: 747 against 1190).
  uint64_t points = 0, coarse = 0;
  for (int s = 0; s < S; ++s) {
    SortSeg& g = h_segs[s];
    if (g.from_cga || g.n_host > kBinMaxPoints) return;
    uint32_t t = 4;
    while (t < kBinMaxBits && ((uint64_t)64 << t) < g.n_host) ++t;
    g.bin_bits = std::min(t, g.bits);
    g.narrow = 3 * g.bits - g.bin_bits <= 30 ? 1u : 0u;
    const uint64_t most = g.narrow ? 4 * bin_cap<uint32_t>() : 4 * bin_cap<unsigned long long>();
    if (g.n_host >> g.bin_bits > most) return;
    if (coarse_build(g)) coarse += g.n_host;
    B.may_split = B.may_split || g.n_host > (g.narrow ? bin_cap<uint32_t>() : bin_cap<unsigned long long>());
    // a job fails by its keys' number or, wide keys only, by its row's parts
    B.may_fall = B.may_fall || g.n_host > kBinRowMax ||
                 (!g.narrow && g.n_host > bin_cap<unsigned long long>());
    B.narrow = B.narrow || g.narrow;
    B.wide = B.wide || !g.narrow;
    points += g.n_host;
  }
  if (2 * coarse > points && !values) return;  // (a batch goes the way of most of its points)
  // partition tiles: enough of them for the SMs, then as many keys a bin as possible
  const uint64_t sms = (uint64_t)device_sm_count();
  B.items = points >= sms * 4 * 16384 ? 16u : (points >= sms * 2 * 8192 ? 8u : 4u);
  uint64_t bins = 0, slots = 0, ptiles = 0, most_big = 0;
  for (int s = 0; s < S; ++s) {
    SortSeg& g = h_segs[s];
    const uint32_t nb = 1u << g.bin_bits, rem = 3 * g.bits - g.bin_bits;
    const uint32_t span = g.narrow ? std::min(32u - rem, kBinMaxBits) : kBinMaxBits;
    // jobs of half a block's capacity, smaller ones while they are too few for the SMs:
    // 100k uniform points, b = 10, 65 us with half a block, 57 with 1024 keys and up,
    // 100k LiDAR points, b = 12, 73 and 59, ten sweeps of 131k, b = 13, 175 and 157
    // (eight jobs an SM, not four: 1M uniform points 84 and 93)
    const uint32_t most_keys = g.narrow ? bin_target<uint32_t>() : bin_target<unsigned long long>();
    const uint32_t target = (uint32_t)std::min<uint64_t>(most_keys, std::max<uint64_t>(1024, points / (4 * sms)));
    g.job_keys = target;
    g.bin_base = (uint32_t)bins;
    g.ptile_base = (uint32_t)ptiles;
    g.job_base = (uint32_t)slots;
    // a job per target's worth of points, two around each larger bin, one per span,
    // and a split bin's slots
    g.job_cap = 7 * (g.n_host / target + 1) + (nb >> span) + 4;
    most_big += g.n_host / (2 * target);
    bins += nb;
    slots += g.job_cap;
    ptiles += (g.n_host + 1024ull * B.items - 1) / (1024ull * B.items);
  }
  const size_t room = (size_t)kMaxPasses * total_tiles * ((size_t)4 << sc.radix_bits);
  char* p = reinterpret_cast<char*>(sc.look);
  auto take = [&](size_t bytes) {
    char* r = p;
    p += align_up(bytes);
    return r;
  };
  B.cnt = reinterpret_cast<uint32_t*>(take(bins * 4));
  B.big = reinterpret_cast<uint2*>(take((most_big + 1) * 8));
  B.zero_words = (uint32_t)((p - reinterpret_cast<char*>(sc.look)) / 4);
  B.cur = reinterpret_cast<uint32_t*>(take(bins * 4));
  B.jobs = reinterpret_cast<uint4*>(take(slots * 16));
  B.info = reinterpret_cast<uint4*>(take(slots * 16));
  B.njobs = reinterpret_cast<uint32_t*>(take((size_t)S * 4));
  // (empty clouds take room here but none in the look-back words: a batch of many goes
  // the general way, with the digits and passes that the caller planned)
  if ((size_t)(p - reinterpret_cast<char*>(sc.look)) > room || slots > 0x7fffffffull) return;
  // the general sort behind the bins has 8-bit digits
  for (int s = 0; s < S; ++s) {
    h_segs[s].passes = radix_passes(h_segs[s].key_bits, 8);
    B.passes = std::max(B.passes, h_segs[s].passes);
  }
  B.ptiles = (uint32_t)ptiles;
  B.slots = (uint32_t)slots;
  B.on = true;
}

template <typename T, bool ROWS>
static void launch_part(int S, const SortScratch& sc, uint32_t stride, cudaStream_t stream) {
  const BinPlan& B = sc.bins;
  T* keys = static_cast<T*>(sc.keys0);
  if (B.items == 16) {
    k_bin_part<T, 16, ROWS><<<B.ptiles, 1024, bin_part_smem<T, 16>(), stream>>>(
        sc.segs, S, B.cur, keys, stride, B.value_in, B.value_rows);
  } else if (B.items == 8) {
    k_bin_part<T, 8, ROWS><<<B.ptiles, 1024, bin_part_smem<T, 8>(), stream>>>(
        sc.segs, S, B.cur, keys, stride, B.value_in, B.value_rows);
  } else {
    k_bin_part<T, 4, ROWS><<<B.ptiles, 1024, bin_part_smem<T, 4>(), stream>>>(
        sc.segs, S, B.cur, keys, stride, B.value_in, B.value_rows);
  }
}

template <typename T, bool ROWS>
static void launch_split(const SortScratch& sc, uint32_t stride, cudaStream_t stream) {
  const BinPlan& B = sc.bins;
  T *k0 = static_cast<T*>(sc.keys0), *k1 = static_cast<T*>(sc.keys1);
  const unsigned clusters = std::max(1u, 3 * (unsigned)device_sm_count() / kBinCluster);
  k_bin_split<T, ROWS><<<clusters * kBinCluster, kBinThreads, 0, stream>>>(
      sc.segs, B.jobs, B.big, k0, k1, stride, B.value_rows, B.value_rows + B.value_in.n);
}

template <typename T>
static void launch_bin_jobs(int S, const SortScratch& sc, uint32_t stride, uint32_t* counter,
                            cudaStream_t stream) {
  const BinPlan& B = sc.bins;
  T *k0 = static_cast<T*>(sc.keys0), *k1 = static_cast<T*>(sc.keys1);
  // (attributes are summed faster by bins than in general, but not a crowded row's)
  const bool values = B.value_rows != nullptr;
  k_bin_scan<T><<<S, 1024, 0, stream>>>(sc.segs, B.cnt, B.cur, B.jobs, B.njobs, B.big, !values);
  if (B.value_rows != nullptr) {
    launch_part<T, true>(S, sc, stride, stream);
    if (B.may_split) launch_split<T, true>(sc, stride, stream);
  } else {
    launch_part<T, false>(S, sc, stride, stream);
    if (B.may_split) launch_split<T, false>(sc, stride, stream);
  }
  const uint32_t blocks = std::min<uint32_t>(B.slots, g_bin_sort_blocks[sizeof(T) / 8]);
  k_bin_sort<T><<<blocks, kBinThreads, bin_sort_smem<T>(), stream>>>(
      sc.segs, S, B.jobs, B.njobs, k0, k1, B.info, counter, B.slots, stride,
      values ? kBinRowMax : kBinSplitMax);
}

template <typename T>
static void launch_bin_write(int S, const SortScratch& sc, uint32_t stride, cudaStream_t stream) {
  const BinPlan& B = sc.bins;
  const T *k0 = static_cast<const T*>(sc.keys0), *k1 = static_cast<const T*>(sc.keys1);
  k_bin_write<T><<<std::min<uint32_t>(B.slots, (uint32_t)device_sm_count() * 8), kThreads, 0,
                   stream>>>(sc.segs, S, B.jobs, B.njobs, k0, k1, B.info, B.slots, stride);
  if (B.value_rows != nullptr) {
    k_bin_values<T><<<std::min<uint32_t>(B.slots, g_bin_values_blocks[sizeof(T) / 8]), kBinThreads,
                      bin_values_smem<T>(), stream>>>(
        sc.segs, B.jobs, B.njobs, k0, k1, B.value_rows, B.value_rows + B.value_in.n, B.info, stride,
        B.value_in, B.values);
    count_launch(1);
  }
}

template <typename K>
static cudaError_t launch_lsd_all(int S, uint32_t total_tiles, const SortScratch& sc,
                                  cudaStream_t stream) {
  const uint32_t words = (uint32_t)((reinterpret_cast<char*>(sc.counters) -
                                     reinterpret_cast<char*>(sc.hist)) / 4);
  k_lsd_all<K><<<g_lsd_blocks[sizeof(K) / 8], kThreads, onesweep_smem<K, kThreads, 8>(), stream>>>(
      sc.segs, S, total_tiles, sc.bins.passes, static_cast<K*>(sc.keys0), static_cast<K*>(sc.keys1),
      sc.hist, sc.look, sc.clook, sc.counters, words);
  return cudaGetLastError();
}

// The build by bins (the plan is laid out, the segment table uploaded).
static cudaError_t run_bins(int S, uint32_t total_tiles, bool key64, const SortScratch& sc,
                            cudaStream_t stream) {
  const cudaError_t ei = init_sort_kernels();
  if (ei != cudaSuccess) return ei;
  const BinPlan& B = sc.bins;
  const uint32_t sms = (uint32_t)device_sm_count(), stride = key64 ? 8u : 4u;
  const uint32_t zb = std::min<uint32_t>((std::max<uint32_t>(B.zero_words, (uint32_t)S) + 255) / 256,
                                         sms * 8);
  k_bin_init<<<zb, 256, 0, stream>>>(sc.segs, S, B.cnt, B.zero_words, sc.counters);
  const uint32_t ctas = std::min<uint32_t>(total_tiles, sms * 4);
  k_bin_hist<<<ctas, kBinThreads, 0, stream>>>(sc.segs, S, total_tiles,
                                               (total_tiles + ctas - 1) / ctas, B.cnt);
  // a launch for each key width in the batch
  if (B.narrow) launch_bin_jobs<uint32_t>(S, sc, stride, sc.counters + kMaxPasses + 1, stream);
  if (B.wide) launch_bin_jobs<unsigned long long>(S, sc, stride, sc.counters + kMaxPasses + 3, stream);
  if (B.narrow) launch_bin_write<uint32_t>(S, sc, stride, stream);
  if (B.wide) launch_bin_write<unsigned long long>(S, sc, stride, stream);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && B.may_fall) {
    e = key64 ? launch_lsd_all<unsigned long long>(S, total_tiles, sc, stream)
              : launch_lsd_all<uint32_t>(S, total_tiles, sc, stream);
  }
  count_launch((B.may_fall ? 3 : 2) + (B.may_split ? 5 : 4) * ((B.narrow ? 1 : 0) + (B.wide ? 1 : 0)));
  // the Value array of a cloud that the general sort had to take
  if (e == cudaSuccess && B.value_rows != nullptr && B.may_fall) {
    e = run_build_values(B.value_out, B.value_in, B.value_rows, B.values, &sc.segs[0].fallback,
                         stream);
  }
  return e;
}

cudaError_t init_sort_kernels() {
  static std::once_flag once;
  static cudaError_t rc = cudaSuccess;
  std::call_once(once, [] {
    const cudaError_t es[] = {
        set_pass_smem<uint32_t, 256, 8>(),           set_pass_smem<uint32_t, 512, 8>(),
        set_pass_smem<uint32_t, 512, 9>(),           set_pass_smem<unsigned long long, 256, 8>(),
        set_pass_smem<unsigned long long, 512, 8>(), set_pass_smem<unsigned long long, 512, 9>()};
    for (cudaError_t e : es) {
      if (e != cudaSuccess && rc == cudaSuccess) rc = e;
    }
    const cudaError_t eb = init_bin_kernels();
    if (eb != cudaSuccess && rc == cudaSuccess) rc = eb;
  });
  return rc;
}

cudaError_t run_radix_passes(int S, uint32_t total_tiles, uint32_t max_passes, bool key64,
                             const SortScratch& sc, cudaStream_t stream) {
  if (total_tiles == 0) return cudaSuccess;
  const cudaError_t ei = init_sort_kernels();
  if (ei != cudaSuccess) return ei;
  if (key64) {
    launch_passes<unsigned long long>(S, total_tiles, max_passes, sc, stream);
  } else {
    launch_passes<uint32_t>(S, total_tiles, max_passes, sc, stream);
  }
  return cudaGetLastError();
}

// Keys and histograms, from points or (walk) from CGAs.
template <typename K>
static void launch_keys(int S, uint32_t total_tiles, bool walk, const SortScratch& sc,
                        cudaStream_t stream) {
  const uint32_t items = walk ? total_tiles * (kTile / kWalkRun) : total_tiles;
  const uint32_t ctas =
      std::min<uint32_t>(items, (uint32_t)device_sm_count() * (walk ? kKeysWalkPerSm : 4));
  const uint32_t per = (items + ctas - 1) / ctas;
  K* k0 = static_cast<K*>(sc.keys0);
  if (walk && sc.radix_bits == 9) {
    k_keys_walk<K, 9><<<ctas, kThreads, 0, stream>>>(sc.segs, S, items, per, k0, sc.hist);
  } else if (walk) {
    k_keys_walk<K, 8><<<ctas, kThreads, 0, stream>>>(sc.segs, S, items, per, k0, sc.hist);
  } else if (sc.radix_bits == 9) {
    k_keys_hist<K, 9><<<ctas, kThreads, 0, stream>>>(sc.segs, S, items, per, k0, sc.hist);
  } else {
    k_keys_hist<K, 8><<<ctas, kThreads, 0, stream>>>(sc.segs, S, items, per, k0, sc.hist);
  }
  count_launch(1);
}

template <typename K>
static cudaError_t launch_pipeline(int S, uint32_t total_tiles, uint32_t max_passes, int levels,
                                   bool walk, const SortScratch& sc, cudaStream_t stream) {
  K* k0 = static_cast<K*>(sc.keys0);
  K* k1 = static_cast<K*>(sc.keys1);
  const cudaError_t ei = init_sort_kernels();
  if (ei != cudaSuccess) return ei;
  launch_keys<K>(S, total_tiles, walk, sc, stream);
  launch_passes<K>(S, total_tiles, max_passes, sc, stream);
  if (levels == 3) {
    k_compact<K, 3><<<total_tiles, kThreads, 0, stream>>>(sc.segs, S, k0, k1, sc.clook,
                                                          sc.counters + kMaxPasses);
  } else {
    k_compact<K, 2><<<total_tiles, kThreads, 0, stream>>>(sc.segs, S, k0, k1, sc.clook,
                                                          sc.counters + kMaxPasses);
  }
  count_launch(1);
  return cudaGetLastError();
}

cudaError_t run_sort_keys_device(int S, uint32_t total_tiles, uint32_t max_passes,
                                 const SortScratch& sc, cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(sc.hist, 0, sc.zero_bytes, stream);
  if (e != cudaSuccess || total_tiles == 0) return e;
  e = init_sort_kernels();
  if (e != cudaSuccess) return e;
  launch_keys<unsigned long long>(S, total_tiles, true, sc, stream);
  launch_passes<unsigned long long>(S, total_tiles, max_passes, sc, stream);
  return cudaGetLastError();
}

cudaError_t run_sort_device(int S, uint32_t total_tiles, uint32_t max_passes, bool key64,
                            int levels, bool from_cga, const SortScratch& sc,
                            cudaStream_t stream) {
  if (sc.bins.on && total_tiles > 0) return run_bins(S, total_tiles, key64, sc, stream);
  cudaError_t e = cudaMemsetAsync(sc.hist, 0, sc.zero_bytes, stream);
  if (e != cudaSuccess) return e;
  k_seg_init<<<(S + 127) / 128, 128, 0, stream>>>(sc.segs, S);
  count_launch(1);
  e = cudaGetLastError();
  if (e != cudaSuccess || total_tiles == 0) return e;
  return key64 ? launch_pipeline<unsigned long long>(S, total_tiles, max_passes, levels, from_cga,
                                                     sc, stream)
               : launch_pipeline<uint32_t>(S, total_tiles, max_passes, levels, from_cga, sc, stream);
}

size_t wait_selftest_bytes() {
  return align_up(sizeof(Header)) + sort_scratch_bytes(2 * kTile, 2, 1, true);
}

// One radix-pass tile that draws tile id 1 of a two-tile segment whose tile 0
// never runs: its look-back word for tile 0 is never published, so the wait
// must give up on its own and record kErrTimeout in *hdr.
cudaError_t run_wait_selftest(void* scratch, cudaStream_t stream) {
  const size_t bytes = wait_selftest_bytes();
  Header* hdr = static_cast<Header*>(scratch);
  const SortScratch sc = sort_scratch_carve(static_cast<char*>(scratch) + align_up(sizeof(Header)),
                                            2 * kTile, 2, 1, true);
  SortSeg seg{};
  seg.n_host = 2 * kTile;
  seg.passes = 1;
  seg.num_tiles = 2;
  seg.out.hdr = hdr;
  const uint32_t first_id = 1;
  cudaError_t e = cudaMemsetAsync(scratch, 0, bytes, stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(sc.segs, &seg, sizeof(SortSeg), cudaMemcpyHostToDevice, stream);
  if (e == cudaSuccess) {
    e = cudaMemcpyAsync(sc.counters, &first_id, sizeof(uint32_t), cudaMemcpyHostToDevice, stream);
  }
  if (e != cudaSuccess) return e;
  e = init_sort_kernels();
  if (e != cudaSuccess) return e;
  k_onesweep<unsigned long long, 512, 8>
      <<<1, 512, onesweep_smem<unsigned long long, 512, 8>(), stream>>>(
      sc.segs, 1, 0, static_cast<const unsigned long long*>(sc.keys0),
      static_cast<unsigned long long*>(sc.keys1), sc.hist, sc.look, sc.counters);
  count_launch(1);
  return cudaGetLastError();
}

cudaError_t run_sort_pipeline(const SortSeg* h_segs, int S, uint32_t total_tiles,
                              uint32_t max_passes, bool key64, const SortScratch& sc,
                              cudaStream_t stream) {
  cudaError_t e = cudaMemcpyAsync(sc.segs, h_segs, sizeof(SortSeg) * S, cudaMemcpyHostToDevice,
                                  stream);
  if (e != cudaSuccess) return e;
  return run_sort_device(S, total_tiles, max_passes, key64, (int)h_segs[0].out.nlevels,
                         h_segs[0].from_cga != 0, sc, stream);
}

}  // namespace libcga
