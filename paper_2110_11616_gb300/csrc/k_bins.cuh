// CGA build by bins: the points are partitioned once by the top bits of their
// voxel keys, and each run of bins is sorted, deduplicated and compacted inside
// one block's shared memory.
//
// An LSD radix sort of the whole cloud reads and writes every 8-byte key once
// per digit and ranks it stably each time (about 40 instructions a key and
// digit; 128 us a pass and 0.94 ms in all for 15M points at b = 12, issue-bound).
// Partitioning by the top bits first needs no stability, so ranks come from
// shared-memory atomics, and what is left of a key (24 bits at b = 12) sorts on
// chip.  The keys cross HBM twice (one write, one read; 4 bytes each when the
// bin and 32 bits give the key) instead of ten times.
//
//   k_bin_init   headers, counters and look-back words
//   k_bin_hist   points per bin (shared-memory counts), non-finite points
//   k_bin_scan   bin offsets; bins grouped into jobs of about half a block's
//                capacity
//   k_bin_part   tiles of points to their bins: counts in shared memory, one
//                global reservation per tile and bin, runs written from a stage
//   k_bin_split  bins beyond a block's capacity (few or none): partitioned once more
//                by their next bits, into jobs of their own
//   k_bin_sort   a job per block: its keys ordered in shared memory, the distinct
//                ones written back with the job's counts
//   k_bin_write  the CGA arrays, a job per block
//   k_bin_values the Value array, a job per block (builds with attributes only)
//
// A bin holds whole x slabs (bin bits <= grid bits) and a job of a split bin whole
// columns, so a job's first key always opens a voxel and a column, and a slab
// unless the job goes on with a slab of its bin.  A bin of more than kBinSplitMax keys (or
// kBinHeavy and a share of the points), or a row of a split (12 more bits) of more than
// kBinRowMax keys that no map takes, marks its segment, which k_lsd_all then sorts the
// general way.  (By the first rule before any job is made: the kernels after k_bin_scan
// then leave the segment alone.  By the second in k_bin_sort, where the segment's keys
// and jobs are all written.)
// Measured on GB300 (us): 15M surface points at b = 12: sort 187, partition 120,
// write 60, histogram 44, split 18, scan 11; the build 954 -> 475.  The job sort is
// bound by the issue of its shared-memory steps, the partition by the latency of one
// wave's loads and reservations.  A 131k LiDAR sweep at b = 16: 113 -> 78 (ten short
// kernels: launch to launch).  LiDAR 1.3M, b = 16: 179 -> 130; uniform 30M, b = 12:
// 1794 -> 721; 10-bit grids, whose bins all have to be split: 2M LiDAR 154 -> 158,
// 15M uniform 747 -> 662, 30M uniform 1377 -> 1368.  A cloud that the general sort
// has to take over pays for the bins too: 1M points in one voxel 140 -> 207.
#pragma once
#include "k_compact.cuh"

namespace libcga {

namespace {

__device__ __forceinline__ int find_seg(const SortSeg* __restrict__ segs, int S, uint32_t t) {
  int lo = 0, hi = S - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (segs[mid].tile_base <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Exclusive scan across a block of TH threads (s_warp: TH/32 words).
template <int TH, typename T>
__device__ __forceinline__ T block_scan_th(T v, T& total, T* s_warp) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T inc = warp_incl_scan(v);
  if (lane == 31) s_warp[w] = inc;
  __syncthreads();
  T before = 0, tot = 0;
#pragma unroll
  for (int i = 0; i < TH / 32; ++i) {
    const T x = s_warp[i];
    if (i < w) before += x;
    tot += x;
  }
  __syncthreads();
  total = tot;
  return before + inc - v;
}

constexpr int kBinThreads = 512;
constexpr int kBinWarps = kBinThreads / 32;
constexpr uint32_t kBinMaxBits = 12;
constexpr uint32_t kBinSplitMax = 1u << 20;   // the most keys of a bin to split
constexpr uint32_t kBinRowMax = 1u << 18;     // the most keys of a row that goes by parts
// A bin that outweighs its cloud (more than this and a 16th of the points): a cluster
// splits it alone, 30 us and 125 for each million of its keys, and most such bins are one
// voxel's, whose row then takes a block as long.  In general 2M points, a quarter of them
// at one point, take 250 us (b = 12; by bins 371) and 276 (b = 16; 415, the general sort
// included), 1M in one voxel 208 and 330; 500k in one slab, though, 201 and 152.
constexpr uint32_t kBinHeavy = (1u << 18) + (1u << 16);
constexpr int kBinWalks = 12;                 // the most passes over such a row
constexpr uint32_t kBinMapBits = 18;          // bits of a key that a block maps
constexpr int kBinCluster = 8;                // blocks that split a bin together
constexpr uint32_t kBigCluster = 1u << 31;    // flag of a bin for a cluster
constexpr uint32_t kBinAlone = 1u << 15;      // keys up to which one block splits a bin
constexpr uint32_t kBinRowBits = 12;          // bits a split goes by
constexpr uint32_t kJobSplit = 1u << 31;      // of a job's first word: a split's job
constexpr uint32_t kJobGoesOn = 1u << 30;     // its first slab has earlier keys

// Job slots of a bin of n keys that is split into jobs of about `target` keys.
__host__ __device__ inline uint32_t split_slots(uint32_t n, uint32_t target) {
  return 3 * (n / target) + 2;
}

// Keys a sorting block holds (two buffers of 32 KB) and what a job aims at.
template <typename T>
constexpr int bin_items() { return sizeof(T) == 4 ? 16 : 8; }
template <typename T>
constexpr uint32_t bin_cap() { return (uint32_t)(kBinThreads * bin_items<T>()); }
template <typename T>
constexpr uint32_t bin_target() { return bin_cap<T>() / 2; }

// Buckets of a block's sort (by the top bits of what its keys differ in), and the
// keys up to which a bucket is ordered by counting.
constexpr uint32_t kBinBucketBits = 12;
constexpr uint32_t kBinBucketMax = 48;
constexpr uint32_t kBinWork = 64;  // comparisons a key, on average, in crowded buckets

// Dynamic shared memory of k_bin_sort: both key buffers, the bucket counts (or the
// warps' digit counts of the LSD passes), a bitmap per warp and the offsets of a
// large job's parts.
template <typename T>
constexpr size_t bin_sort_smem() {
  return 2 * sizeof(T) * (size_t)bin_cap<T>() + 2 * ((1u << kBinBucketBits) + 4) * sizeof(uint32_t) +
         (size_t)kBinWarps * ((1u << kBinBucketBits) / 8);
}
// Of k_bin_part: the staged keys, the tile's counts and output offsets per bin.
template <typename T, int IT>
constexpr size_t bin_part_smem() {
  return sizeof(T) * 1024 * IT + 2 * sizeof(uint32_t) * (1u << kBinMaxBits);
}

__global__ void k_bin_init(SortSeg* segs, int S, uint32_t* zero, uint32_t words,
                           uint32_t* counters) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (uint32_t s = i; s < (uint32_t)S; s += stride) {
    const Levels& o = segs[s].out;
    o.hdr->cnt[0] = 0;
    o.hdr->cnt[1] = 0;
    o.hdr->cnt[2] = 0;
    o.hdr->err = 0;
    o.ptr1[0] = 0;
    o.ptr2[0] = 0;
    segs[s].fallback = 0;
  }
  for (uint32_t w = i; w < words; w += stride) zero[w] = 0;
  if (i < kCounterWords) counters[i] = 0;
}

// Four consecutive points (the first a multiple of four) by three 16-byte loads
// where the array allows, else by single loads; points at or past n read as 0.
__device__ __forceinline__ void load_points(const float* __restrict__ xyz, bool vec, uint32_t i,
                                            uint32_t n, float (&p)[12]) {
  if (vec && i + 4 <= n) {
    const float4* q = reinterpret_cast<const float4*>(xyz + 3 * (size_t)i);
    const float4 a = __ldg(q), b = __ldg(q + 1), c = __ldg(q + 2);
    p[0] = a.x; p[1] = a.y; p[2] = a.z; p[3] = a.w;
    p[4] = b.x; p[5] = b.y; p[6] = b.z; p[7] = b.w;
    p[8] = c.x; p[9] = c.y; p[10] = c.z; p[11] = c.w;
  } else {
#pragma unroll
    for (uint32_t k = 0; k < 12; ++k) {
      p[k] = i + k / 3 < n ? __ldg(xyz + 3 * (size_t)i + k) : 0.0f;
    }
  }
}

__device__ __forceinline__ unsigned long long seg_key(const SortSeg& sg, const float* p, bool& ok) {
  unsigned long long key;
  ok = point_key<unsigned long long>(p[0], p[1], p[2], sg.has_x != 0, sg.X, sg.scale, sg.off,
                                     sg.bits, key);
  return key;
}

// A segment's part of a key buffer: its first slot counted in the buffer's own keys
// (of `stride` bytes, 8 when any key of the batch has more than 32 bits).
template <typename T>
__device__ __forceinline__ T* seg_keys(T* buf, const SortSeg& sg, uint32_t stride) {
  return buf + sg.key_base * (stride / sizeof(T));
}
template <typename T>
__device__ __forceinline__ const T* seg_keys(const T* buf, const SortSeg& sg, uint32_t stride) {
  return buf + sg.key_base * (stride / sizeof(T));
}

__device__ __forceinline__ bool points_vec(const SortSeg& sg) {
  return (reinterpret_cast<uintptr_t>(sg.xyz) & 15u) == 0;
}

__global__ void __launch_bounds__(kBinThreads, 4) k_bin_hist(const SortSeg* __restrict__ segs, int S,
                                                             uint32_t total_tiles,
                                                             uint32_t tiles_per_cta,
                                                             uint32_t* __restrict__ cnt) {
  __shared__ uint32_t s_hist[1 << kBinMaxBits];
  __shared__ uint32_t s_err;
  const uint32_t tid = threadIdx.x;
  const uint32_t t0 = blockIdx.x * tiles_per_cta, t1 = min(t0 + tiles_per_cta, total_tiles);
  if (t0 >= t1) return;
  for (uint32_t i = tid; i < (1u << kBinMaxBits); i += kBinThreads) s_hist[i] = 0;
  if (tid == 0) s_err = 0;
  __syncthreads();
  for (uint32_t t = t0; t < t1;) {
    // the block's run of tiles of one segment
    const int s = find_seg(segs, S, t);
    const SortSeg& sg = segs[s];
    const uint32_t te = min(t1, sg.tile_base + sg.num_tiles);
    const uint32_t i0 = (t - sg.tile_base) * kTile, i1 = min(sg.n_host, (te - sg.tile_base) * kTile);
    const uint32_t shift = 3 * sg.bits - sg.bin_bits;
    const bool vec = points_vec(sg);
    bool bad = false;
    for (uint32_t i = i0 + 4 * tid; i < i1; i += 4 * kBinThreads) {
      float p[12];
      load_points(sg.xyz, vec, i, i1, p);
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) {
        bool ok;
        const unsigned long long key = seg_key(sg, p + 3 * k, ok);
        if (i + k < i1) {
          bad = bad || !ok;
          atomicAdd(&s_hist[(uint32_t)(key >> shift)], 1u);
        }
      }
    }
    if (bad) atomicOr(&s_err, kErrNonfinite);
    __syncthreads();
    for (uint32_t i = tid; i < (1u << sg.bin_bits); i += kBinThreads) {
      const uint32_t v = s_hist[i];
      if (v) atomicAdd(cnt + sg.bin_base + i, v);
      s_hist[i] = 0;
    }
    if (tid == 0 && s_err) {
      atomicOr(&sg.out.hdr->err, s_err);
      s_err = 0;
    }
    __syncthreads();
    t = te;
  }
}

// One block per segment: offsets of its bins and its jobs.  A job is {first bin and
// flags, bins, first key, keys}; a bin beyond a block's capacity gets slots for its
// split, and a word {segment, first slot} in `big` (big[0]: how many; kBigCluster: a
// bin for a cluster of blocks).
template <typename T>
__global__ void __launch_bounds__(1024) k_bin_scan(SortSeg* segs,
                                                   const uint32_t* __restrict__ cnt,
                                                   uint32_t* __restrict__ cur,
                                                   uint4* __restrict__ jobs,
                                                   uint32_t* __restrict__ njobs,
                                                   uint2* __restrict__ big, bool heavy) {
  constexpr uint32_t PER = (1u << kBinMaxBits) / 1024;
  __shared__ uint32_t s_scan[32], s_start[(1u << kBinMaxBits) + 1], s_next[32];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
  SortSeg& sg = segs[blockIdx.x];
  if (sg.narrow != (sizeof(T) == 4 ? 1u : 0u)) return;
  const uint32_t bins = 1u << sg.bin_bits, target = sg.job_keys;
  uint32_t c[PER], sum = 0, tot = 0;
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    const uint32_t b = tid * PER + i;
    c[i] = b < bins ? cnt[sg.bin_base + b] : 0u;
    sum += c[i];
  }
  uint32_t run = block_scan_th<1024>(sum, tot, s_scan);
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    const uint32_t b = tid * PER + i;
    if (b < bins) {
      s_start[b] = run;
      cur[sg.bin_base + b] = run;
    }
    run += c[i];
  }
  if (tid == 0) s_start[bins] = tot;
  __syncthreads();
  // a bin opens a job at the target's multiples, next to a bin beyond the target
  // and at the reach of a T (span bins)
  const uint32_t rem = 3 * sg.bits - sg.bin_bits;
  const uint32_t span_bits = min(8 * (uint32_t)sizeof(T) - rem, kBinMaxBits);
  uint32_t nsub[PER], nj = 0, open = 0;
  const uint32_t most = heavy ? min(kBinSplitMax, kBinHeavy + s_start[bins] / 16) : kBinSplitMax;
  bool over = false;
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    const uint32_t b = tid * PER + i;
    nsub[i] = 0;
    if (b >= bins) continue;
    const uint32_t st = s_start[b], n = s_start[b + 1] - st;
    const uint32_t pst = b > 0 ? s_start[b - 1] : 0u;
    const bool large = n > target, plarge = b > 0 && st - pst > target;
    if (b == 0 || large || plarge || st / target != pst / target ||
        (b & ((1u << span_bits) - 1u)) == 0u) {
      nsub[i] = 1;
      if (n > most) {
        over = true;
      } else if (n > bin_cap<T>()) {
        nsub[i] = split_slots(n, target);
      }
      nj += nsub[i];
      open |= 1u << i;
    }
  }
  if (__syncthreads_or(over)) {
    // a marked segment has no jobs: its points are not partitioned and its larger bins
    // not split, so there are no keys, and no split's jobs, for k_bin_sort to read
    if (tid == 0) {
      sg.fallback = 1;
      njobs[blockIdx.x] = 0;
    }
    return;
  }
  uint32_t j = block_scan_th<1024>(nj, tot, s_scan);
  const uint32_t all = min(tot, sg.job_cap);
  // the first job-opening bin after this thread's (bins: none): a suffix minimum
  const uint32_t mine = open ? tid * PER + (uint32_t)__ffs((int)open) - 1u : bins;
  uint32_t after = __shfl_down_sync(0xffffffffu, mine, 1);
  if (lane == 31) after = bins;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_down_sync(0xffffffffu, after, o);
    if (lane + o < 32) after = min(after, x);
  }
  if (lane == 0) s_next[w] = min(mine, after);
  __syncthreads();
  for (uint32_t x = w + 1; x < 32; ++x) after = min(after, s_next[x]);
  if (nj > 0) {
#pragma unroll
    for (int i = (int)PER - 1; i >= 0; --i) {
      if (nsub[i] == 0) continue;
      const uint32_t b = tid * PER + (uint32_t)i;
      nj -= nsub[i];
      const uint32_t at = j + nj;
      if (at + nsub[i] <= sg.job_cap) {
        const uint32_t st = s_start[b];
        jobs[sg.job_base + at] = make_uint4(b, after - b, st, s_start[after] - st);
        if (nsub[i] > 1) {
          const uint32_t cluster = s_start[after] - st > kBinAlone ? kBigCluster : 0u;
          big[atomicAdd(&big[0].x, 1u) + 1] = make_uint2(blockIdx.x | cluster, sg.job_base + at);
        }
      }
      after = b;
    }
  }
  if (tid == 0) njobs[blockIdx.x] = all;
}

// What the Value array needs of each of four consecutive points from i (a multiple
// of four): its row, a channel a byte, or its index where the first point counts.
__device__ __forceinline__ void load_rows(const ValueInput& in, uint32_t i, uint32_t n, uint32_t* r) {
  const uint32_t C = in.channels;
  if (in.policy == kValueFirst) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) r[k] = i + k;
    return;
  }
  const uint8_t* p = in.attr + (size_t)i * C;
  if (i + 4 <= n && (reinterpret_cast<uintptr_t>(in.attr) & 3u) == 0) {
    const uint32_t* q = reinterpret_cast<const uint32_t*>(p);
    uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      if (k < C) w[k] = __ldg(q + k);
    }
    if (C == 1) {
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) r[k] = (w[0] >> (8 * k)) & 0xffu;
    } else if (C == 2) {
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) r[k] = (w[k >> 1] >> (16 * (k & 1))) & 0xffffu;
    } else if (C == 3) {
      r[0] = w[0] & 0xffffffu;
      r[1] = __funnelshift_r(w[0], w[1], 24) & 0xffffffu;
      r[2] = __funnelshift_r(w[1], w[2], 16) & 0xffffffu;
      r[3] = w[2] >> 8;
    } else {
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) r[k] = w[k];
    }
    return;
  }
#pragma unroll
  for (uint32_t k = 0; k < 4; ++k) {
    r[k] = 0;
    for (uint32_t c = 0; c < C && i + k < n; ++c) r[k] |= (uint32_t)__ldg(p + k * C + c) << (8 * c);
  }
}

// Tiles of 1024 * IT points into their bins; with ROWS each point's load_rows word
// goes to the same place of `rows`.
template <typename T, int IT, bool ROWS>
__global__ void __launch_bounds__(1024) k_bin_part(const SortSeg* __restrict__ segs, int S,
                                                   uint32_t* __restrict__ cur, T* __restrict__ keys,
                                                   uint32_t stride, ValueInput in,
                                                   uint32_t* __restrict__ rows) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  T* s_key = reinterpret_cast<T*>(s_raw);
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(s_raw + sizeof(T) * 1024 * IT);
  uint32_t* s_off = s_cnt + (1u << kBinMaxBits);
  __shared__ uint32_t s_scan[32];
  __shared__ uint16_t s_bin[1024 * IT];  // bin of each staged key
  constexpr uint32_t PER = (1u << kBinMaxBits) / 1024;
  const uint32_t tid = threadIdx.x;
  int lo = 0, hi = S - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (segs[mid].ptile_base <= blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const SortSeg& sg = segs[lo];
  const uint32_t i0 = (blockIdx.x - sg.ptile_base) * (1024u * IT);
  if (i0 >= sg.n_host || sg.narrow != (sizeof(T) == 4 ? 1u : 0u) || sg.fallback) return;
  const uint32_t i1 = min(i0 + 1024u * IT, sg.n_host);
  const uint32_t bins = 1u << sg.bin_bits, shift = 3 * sg.bits - sg.bin_bits;
  const bool vec = points_vec(sg);
  for (uint32_t b = tid; b < (1u << kBinMaxBits); b += 1024) s_cnt[b] = 0;
  __syncthreads();
  T key[IT];
  uint32_t br[IT];  // bin << 16 | rank in the tile's bin
#pragma unroll
  for (int q = 0; q < IT / 4; ++q) {
    const uint32_t i = i0 + 4 * (tid + 1024u * q);
    float p[12];
    load_points(sg.xyz, vec, i, i1, p);
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      bool ok;
      const unsigned long long v = seg_key(sg, p + 3 * k, ok);
      const uint32_t b = (uint32_t)(v >> shift);
      key[4 * q + k] = (T)v;
      br[4 * q + k] = 0xffffffffu;
      if (i + k < i1) br[4 * q + k] = b << 16 | atomicAdd(&s_cnt[b], 1u);
    }
  }
  __syncthreads();
  uint32_t c[PER], sum = 0, tot = 0;
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    c[i] = s_cnt[tid * PER + i];
    sum += c[i];
  }
  uint32_t run = block_scan_th<1024>(sum, tot, s_scan);
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    const uint32_t b = tid * PER + i;
    s_cnt[b] = run;  // the bin's first staged key
    if (c[i] && b < bins) s_off[b] = atomicAdd(cur + sg.bin_base + b, c[i]) - run;
    run += c[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    if (br[i] != 0xffffffffu) {
      const uint32_t at = s_cnt[br[i] >> 16] + (br[i] & 0xffffu);
      s_key[at] = key[i];
      s_bin[at] = (uint16_t)(br[i] >> 16);
    }
  }
  __syncthreads();
  T* out = seg_keys(keys, sg, stride);
  for (uint32_t e = tid; e < i1 - i0; e += 1024) {
    const uint32_t at = s_off[s_bin[e]] + e;
    if (at < sg.n_host) out[at] = s_key[e];
  }
  if constexpr (ROWS) {
    __syncthreads();
    uint32_t* s_row = reinterpret_cast<uint32_t*>(s_raw);
#pragma unroll
    for (int q = 0; q < IT / 4; ++q) {
      const uint32_t i = i0 + 4 * (tid + 1024u * q);
      uint32_t r[4] = {0, 0, 0, 0};
      if (i < i1) load_rows(in, i, i1, r);
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) {
        const uint32_t v = br[4 * q + k];
        if (v != 0xffffffffu) s_row[s_cnt[v >> 16] + (v & 0xffffu)] = r[k];
      }
    }
    __syncthreads();
    for (uint32_t e = tid; e < i1 - i0; e += 1024) {
      const uint32_t at = s_off[s_bin[e]] + e;
      if (at < sg.n_host) rows[at] = s_row[e];
    }
  }
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

// The shared-memory word `p` of block `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_word(const uint32_t* p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}

__device__ __forceinline__ uint32_t cluster_load(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

__device__ __forceinline__ void cluster_store(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Bins beyond a block's capacity: their keys partitioned by their next bits (whole
// columns) into `out`, at the same places of the segment, and their jobs.  A block
// takes a bin of up to kBinAlone keys, a cluster of blocks a larger one, a part of its
// keys each: the blocks' counts of a row become their offsets in it through the
// cluster's shared memory (block r sums the r-th part of the rows).  The exchange costs
// a bin about 30 us, a block about 15 us for each 15k keys: 1024 bins of 15k keys (15M
// points, b = 10) took the build from 660 to 1190 us with a cluster each; a bin of 173k
// keys (1.3M LiDAR points, b = 10), left to the general sort while a block split every
// bin, cost 313 us there.
template <typename T, bool ROWS>
__global__ void __cluster_dims__(kBinCluster, 1, 1) __launch_bounds__(kBinThreads)
    k_bin_split(const SortSeg* __restrict__ segs, uint4* __restrict__ jobs,
                const uint2* __restrict__ big, const T* __restrict__ keys, T* __restrict__ out,
                uint32_t stride, const uint32_t* __restrict__ rows_in,
                uint32_t* __restrict__ rows_out) {
  constexpr uint32_t R = 1u << kBinRowBits, PER = R / kBinThreads;
  __shared__ uint32_t s_cnt[R], s_tot[R / kBinCluster], s_pre[R + 1], s_scan[kBinWarps],
      s_next[kBinWarps];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
  const uint32_t nbig = big[0].x;
  // the bins that a block takes alone, then those for the cluster
  const uint32_t n1 = blockIdx.x < nbig ? (nbig - 1 - blockIdx.x) / gridDim.x + 1 : 0u;
  const uint32_t cl = blockIdx.x / kBinCluster, ncl = gridDim.x / kBinCluster;
  const uint32_t n2 = cl < nbig ? (nbig - 1 - cl) / ncl + 1 : 0u;
  for (uint32_t i = 0; i < n1 + n2; ++i) {
    const bool alone = i < n1;
    const uint2 B = big[1 + (alone ? blockIdx.x + i * gridDim.x : cl + (i - n1) * ncl)];
    const SortSeg& sg = segs[B.x & ~kBigCluster];
    if (((B.x & kBigCluster) == 0u) != alone) continue;
    if (sg.narrow != (sizeof(T) == 4 ? 1u : 0u) || sg.fallback) continue;
    const uint32_t rank = alone ? 0u : cluster_rank(), parts = alone ? 1u : kBinCluster;
    const uint4 job = jobs[B.y];
    const uint32_t b = sg.bits, rem = 3 * b - sg.bin_bits, N = job.w, target = sg.job_keys;
    const uint32_t rb = min(kBinRowBits, rem - b), shift = rem - rb, rows = 1u << rb;
    // rows of one slab: those that share the key's x bits below the bin's
    const uint32_t xb = min(rb, b - sg.bin_bits), slab = rb - xb;
    const T org = (T)((unsigned long long)job.x << rem);
    const T* src = seg_keys(keys, sg, stride) + job.z;
    T* dst = seg_keys(out, sg, stride) + job.z;
    const uint32_t part = (N + parts - 1) / parts;
    const uint32_t e_lo = min(N, part * rank), e_hi = min(N, e_lo + part);
    for (uint32_t r = tid; r < R; r += kBinThreads) s_cnt[r] = 0;
    __syncthreads();
    for (uint32_t e0 = e_lo + tid; e0 < e_hi; e0 += 8 * kBinThreads) {
      T v[8];
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) {
        const uint32_t e = e0 + k * kBinThreads;
        v[k] = e < e_hi ? __ldg(src + e) : (T)0;
      }
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) {
        if (e0 + k * kBinThreads < e_hi) {
          atomicAdd(s_cnt + (uint32_t)((T)(v[k] - org) >> shift), 1u);
        }
      }
    }
    uint32_t c[PER], sum = 0, tot;
    if (alone) {
      __syncthreads();
#pragma unroll
      for (uint32_t k = 0; k < PER; ++k) {
        c[k] = s_cnt[tid * PER + k];
        s_cnt[tid * PER + k] = 0;
        sum += c[k];
      }
    } else {
      // the cluster's counts: this block's rows become the blocks' offsets in the row
      cluster_sync();
      for (uint32_t r = tid; r < R / kBinCluster; r += kBinThreads) {
        uint32_t a[kBinCluster], v[kBinCluster], run = 0;
#pragma unroll
        for (uint32_t k = 0; k < kBinCluster; ++k) {
          a[k] = cluster_word(s_cnt + rank * (R / kBinCluster) + r, k);
          v[k] = cluster_load(a[k]);
        }
#pragma unroll
        for (uint32_t k = 0; k < kBinCluster; ++k) {
          cluster_store(a[k], run);
          run += v[k];
        }
        s_tot[r] = run;
      }
      cluster_sync();
#pragma unroll
      for (uint32_t k = 0; k < PER; ++k) {
        const uint32_t r = tid * PER + k;
        c[k] = cluster_load(cluster_word(s_tot + r % (R / kBinCluster), r / (R / kBinCluster)));
        sum += c[k];
      }
    }
    uint32_t run = block_scan_th<kBinThreads>(sum, tot, s_scan);
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) {
      s_pre[tid * PER + k] = run;
      s_cnt[tid * PER + k] += run;  // this block's next free place in the row
      run += c[k];
    }
    if (tid == 0) s_pre[R] = N;
    __syncthreads();
    // rows that open a job: at the target's multiples and around larger rows
    uint32_t open = 0, nj = 0;
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) {
      const uint32_t r = tid * PER + k;
      const uint32_t p = s_pre[r], q = r > 0 ? s_pre[r - 1] : 0u;
      if (r < rows && (r == 0 || c[k] > target || p - q > target ||
                       p / target != q / target)) {
        open |= 1u << k;
        ++nj;
      }
    }
    const uint32_t mine = open ? tid * PER + (uint32_t)__ffs((int)open) - 1u : rows;
    uint32_t after = __shfl_down_sync(0xffffffffu, mine, 1);
    if (lane == 31) after = rows;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_down_sync(0xffffffffu, after, o);
      if (lane + o < 32) after = min(after, x);
    }
    if (lane == 0) s_next[w] = min(mine, after);
    uint32_t j = block_scan_th<kBinThreads>(nj, tot, s_scan);
    for (uint32_t x = w + 1; x < (uint32_t)kBinWarps; ++x) after = min(after, s_next[x]);
    // the first block writes the jobs
    const uint32_t slots = rank == 0 ? split_slots(N, target) : 0u;
#pragma unroll
    for (int k = (int)PER - 1; k >= 0; --k) {
      if (!((open >> k) & 1u)) continue;
      const uint32_t r = tid * PER + (uint32_t)k, p = s_pre[r];
      --nj;
      // the row of the job's first key: the last one that starts at p
      uint32_t lo = r, hi = rows - 1;
      while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (s_pre[mid] <= p) lo = mid; else hi = mid - 1;
      }
      const bool on = p > s_pre[(lo >> slab) << slab];
      if (j + nj < slots) {
        jobs[B.y + j + nj] = make_uint4(job.x | kJobSplit | (on ? kJobGoesOn : 0u), 1u, job.z + p,
                                        (after == rows ? N : s_pre[after]) - p);
      }
      after = r;
    }
    for (uint32_t x = tot + tid; x < slots; x += kBinThreads) {
      jobs[B.y + x] = make_uint4(job.x | kJobSplit, 1u, job.z, 0u);
    }
    for (uint32_t e0 = e_lo + tid; e0 < e_hi; e0 += 8 * kBinThreads) {
      T v[8];
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) {
        const uint32_t e = e0 + k * kBinThreads;
        v[k] = e < e_hi ? __ldg(src + e) : (T)0;
      }
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) {
        if (e0 + k * kBinThreads < e_hi) {
          const uint32_t at = atomicAdd(&s_cnt[(uint32_t)((T)(v[k] - org) >> shift)], 1u);
          dst[at] = v[k];
          if constexpr (ROWS) rows_out[job.z + at] = __ldg(rows_in + job.z + e0 + k * kBinThreads);
        }
      }
    }
    // the counts are read and written no more
    if (alone) {
      __syncthreads();
    } else {
      cluster_sync();
    }
  }
}

struct BinSortSmem {
  uint32_t scan[kBinWarps];
  uint32_t off[256];
  uint32_t wcnt[kBinWarps][3];
  uint32_t tot[6];
  uint32_t n;
  uint32_t slot;
  int seg;
  uint32_t nbig;
  uint32_t work;
  uint16_t big[(2 * bin_cap<uint32_t>()) / kBinBucketMax];  // buckets beyond kBinBucketMax
};

// Stable LSD sort of a[0, n) on the low `bits` bits by the whole block (a and b
// of bin_cap entries); returns the buffer that holds the result.
template <typename T>
__device__ __forceinline__ T* bin_block_sort(T* a, T* b, uint32_t n, uint32_t bits,
                                             uint16_t (*wh)[256], BinSortSmem& sm) {
  constexpr int IT = bin_items<T>();
  const uint32_t tid = threadIdx.x, lane = tid & 31u, w = tid >> 5, full = 0xffffffffu;
  const uint32_t ltm = lanemask_lt();
  const uint32_t per = (n + kBinThreads - 1) / kBinThreads;
  for (uint32_t shift = 0; shift < bits; shift += 8) {
    for (uint32_t i = tid; i < kBinWarps * 128; i += kBinThreads) {
      reinterpret_cast<uint32_t*>(wh)[i] = 0;
    }
    __syncthreads();
    T k[IT];
    uint32_t dr[IT];  // digit << 16 | rank in the warp, all ones: no key
#pragma unroll
    for (int i = 0; i < IT; ++i) {
      dr[i] = full;
      k[i] = 0;
      if ((uint32_t)i < per) {
        const uint32_t e = w * 32u * per + i * 32u + lane;
        const bool v = e < n;
        if (v) k[i] = a[e];
        const uint32_t d = (uint32_t)(k[i] >> shift) & 255u;
        uint32_t peers = __ballot_sync(full, v);
        if (!v) peers = ~peers;
#pragma unroll
        for (int bit = 0; bit < 8; ++bit) {
          const uint32_t vote = __ballot_sync(full, (d >> bit) & 1u);
          peers &= ((d >> bit) & 1u) ? vote : ~vote;
        }
        const uint32_t base = v ? wh[w][d] : 0u;
        __syncwarp();
        if (v && lane == (uint32_t)__ffs((int)peers) - 1u) wh[w][d] = (uint16_t)(base + __popc(peers));
        __syncwarp();
        if (v) dr[i] = d << 16 | (base + __popc(peers & ltm));
      }
    }
    __syncthreads();
    uint32_t total = 0, all;
    if (tid < 256) {
#pragma unroll
      for (int x = 0; x < kBinWarps; ++x) {
        const uint32_t c = wh[x][tid];
        wh[x][tid] = (uint16_t)total;
        total += c;
      }
    }
    const uint32_t first = block_scan_th<kBinThreads>(total, all, sm.scan);
    if (tid < 256) sm.off[tid] = first;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < IT; ++i) {
      if (dr[i] != full) {
        const uint32_t d = dr[i] >> 16;
        b[sm.off[d] + wh[w][d] + (dr[i] & 0xffffu)] = k[i];
      }
    }
    __syncthreads();
    T* t = a;
    a = b;
    b = t;
  }
  return a;
}

// a[0, n) in ascending order by the whole block: keys that differ in their low
// `bits` bits only.  A counting sort by the top 12 of those bits leaves buckets of
// about a key each (ranks by shared-memory atomics: order inside a bucket is
// free), and every key then counts the smaller ones of its bucket: about 60
// instructions a key against 170 of three stable 8-bit passes, and a third of
// their barriers.  A bucket of more than kBinBucketMax keys (duplicates of one
// voxel, a dense column) goes through a warp's bitmap of what is left of its keys:
// its distinct keys in order, the rest of its places filled with the last of them.
// Where that takes more than 12 bits, the keys of such buckets are counted like the
// others, or the whole block falls back to the stable passes when that means more than
// kBinWork comparisons a key (by one bucket's size, 384 keys, instead: ten LiDAR sweeps
// of 131k at b = 13 157 us against 134, 15M surface points at b = 13 534 against 510;
// limits of 32 to 96 are within 1% of each other, 160 and none slower).
template <typename T>
__device__ __forceinline__ T* bin_block_order(T* a, T* b, uint32_t n, uint32_t bits, uint32_t* cnt,
                                              BinSortSmem& sm) {
  constexpr int IT = bin_items<T>();
  constexpr uint32_t NB = 1u << kBinBucketBits, PER = NB / kBinThreads;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, w = tid >> 5, full = 0xffffffffu;
  const uint32_t H = min(bits, kBinBucketBits), sh = bits - H, m = (1u << H) - 1u;
#pragma unroll
  for (uint32_t i = 0; i < PER / 4; ++i) {
    reinterpret_cast<uint4*>(cnt)[tid + kBinThreads * i] = make_uint4(0, 0, 0, 0);
  }
  if (tid == 0) sm.nbig = sm.work = 0;
  __syncthreads();
  T k[IT];
  uint32_t r[IT];
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    const uint32_t e = tid + (uint32_t)kBinThreads * i;
    k[i] = 0;
    r[i] = 0;
    if (e < n) {
      k[i] = a[e];
      r[i] = atomicAdd(cnt + ((uint32_t)(k[i] >> sh) & m), 1u);
    }
  }
  __syncthreads();
  uint32_t c[PER], sum = 0, all;
#pragma unroll
  for (uint32_t i = 0; i < PER; i += 4) {
    const uint4 q = reinterpret_cast<const uint4*>(cnt)[(tid * PER + i) / 4];
    c[i] = q.x;
    c[i + 1] = q.y;
    c[i + 2] = q.z;
    c[i + 3] = q.w;
  }
  uint32_t work = 0;  // comparisons in the buckets that no bitmap takes
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    sum += c[i];
    if (c[i] > kBinBucketMax) {
      if (sh <= kBinBucketBits) {
        sm.big[atomicAdd(&sm.nbig, 1u)] = (uint16_t)(tid * PER + i);
      } else {
        work += c[i] * c[i];
      }
    }
  }
  work = __reduce_add_sync(full, work);
  if (lane == 0 && work) atomicAdd(&sm.work, work);
  __syncthreads();
  if (sm.work > kBinWork * n) {
    return bin_block_sort<T>(a, b, n, bits, reinterpret_cast<uint16_t (*)[256]>(cnt), sm);
  }
  uint32_t run = block_scan_th<kBinThreads>(sum, all, sm.scan);
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    const uint32_t x = c[i];
    c[i] = run;
    run += x;
  }
#pragma unroll
  for (uint32_t i = 0; i < PER; i += 4) {
    reinterpret_cast<uint4*>(cnt)[(tid * PER + i) / 4] = make_uint4(c[i], c[i + 1], c[i + 2], c[i + 3]);
  }
  if (tid == 0) cnt[NB] = n;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    const uint32_t e = tid + (uint32_t)kBinThreads * i;
    if (e < n) b[cnt[(uint32_t)(k[i] >> sh) & m] + r[i]] = k[i];
  }
  __syncthreads();
  for (uint32_t e = tid; e < n; e += kBinThreads) {
    const T key = b[e];
    const uint32_t d = (uint32_t)(key >> sh) & m;
    const uint32_t s = cnt[d], f = cnt[d + 1];
    if (f - s > kBinBucketMax && sh <= kBinBucketBits) continue;  // by a bitmap
    uint32_t at = s;
    for (uint32_t x = s; x < f; ++x) {
      const T o = b[x];
      at += o < key || (o == key && x < e) ? 1u : 0u;
    }
    a[at] = key;
  }
  uint32_t* map = cnt + NB + 4 + w * (NB / 32);
  for (uint32_t q = w; q < sm.nbig; q += kBinWarps) {
    constexpr uint32_t WPL = NB / 1024;  // words of the bitmap per lane
    const uint32_t d = sm.big[q], s = cnt[d], f = cnt[d + 1];
    const T top = (b[s] >> sh) << sh;
#pragma unroll
    for (uint32_t i = 0; i < WPL; ++i) map[lane * WPL + i] = 0;
    __syncwarp();
    for (uint32_t e = s + lane; e < f; e += 32) {
      const uint32_t z = (uint32_t)(b[e] - top);
      atomicOr(map + (z >> 5), 1u << (z & 31u));
    }
    __syncwarp();
    uint32_t word[WPL], n1 = 0;
#pragma unroll
    for (uint32_t i = 0; i < WPL; ++i) {
      word[i] = map[lane * WPL + i];
      n1 += (uint32_t)__popc(word[i]);
    }
    const uint32_t inc = warp_incl_scan(n1);
    uint32_t at = s + inc - n1;
    uint32_t hi = 0;  // the lane's greatest z + 1
#pragma unroll
    for (uint32_t i = 0; i < WPL; ++i) {
      for (uint32_t x = word[i]; x != 0u; x &= x - 1u) {
        const uint32_t z = (lane * WPL + i) * 32 + (uint32_t)__ffs((int)x) - 1u;
        a[at++] = top + (T)z;
        hi = z + 1;
      }
    }
    hi = __reduce_max_sync(full, hi);
    const uint32_t used = __shfl_sync(full, inc, 31);
    for (uint32_t e = s + used + lane; e < f; e += 32) a[e] = top + (T)(hi - 1);
    __syncwarp();
  }
  __syncthreads();
  return a;
}

// The distinct keys of the sorted a[0, n) to b, in order; returns their number.
template <typename T>
__device__ __forceinline__ uint32_t bin_block_unique(const T* a, T* b, uint32_t n,
                                                     BinSortSmem& sm) {
  constexpr int IT = bin_items<T>();
  const uint32_t per = (n + kBinThreads - 1) / kBinThreads;
  const uint32_t e0 = threadIdx.x * per;
  uint32_t c = 0, all;
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    const uint32_t e = e0 + i;
    if ((uint32_t)i < per && e < n && (e == 0 || a[e] != a[e - 1])) ++c;
  }
  uint32_t at = block_scan_th<kBinThreads>(c, all, sm.scan);
#pragma unroll
  for (int i = 0; i < IT; ++i) {
    const uint32_t e = e0 + i;
    if ((uint32_t)i < per && e < n && (e == 0 || a[e] != a[e - 1])) b[at++] = a[e];
  }
  __syncthreads();
  return all;
}

// Jobs by the resident blocks.  A job's distinct keys, in order, go to the places
// of its keys in the other buffer (a split's jobs read from that one and write to
// the first), its counts of voxels, columns and slabs to info: {first place,
// voxels, columns, slabs}.  Nothing waits for another job here: writing the CGA
// from this kernel, behind a look-back over the jobs, held finished blocks up for
// more than half the time (26 of 44 us a job) whenever one job was slower than its
// successors.  A row of a split with more keys than the block holds goes through a
// map of the bits that are left (narrow keys), or by parts that fit and maps of the
// parts that don't: duplicates cost a read each (100k points, nine tenths of them in
// one voxel, b = 12: 98 -> 85 us; a tenth of a 131k sweep at one point, b = 16:
// 112 -> 93).
template <typename T>
__global__ void __launch_bounds__(kBinThreads, 2)
    k_bin_sort(SortSeg* segs, int S, const uint4* __restrict__ jobs,
               const uint32_t* __restrict__ njobs, T* keys0, T* keys1, uint4* __restrict__ info,
               uint32_t* counter, uint32_t total_slots, uint32_t stride, uint32_t map_most) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  __shared__ BinSortSmem sm;
  __shared__ uint32_t s_cnt[2];
  constexpr int IT = bin_items<T>();
  constexpr uint32_t CAP = bin_cap<T>();
  T* const buf0 = reinterpret_cast<T*>(s_raw);
  T* const buf1 = buf0 + CAP;
  uint32_t* cnt = reinterpret_cast<uint32_t*>(buf1 + CAP);
  const uint32_t tid = threadIdx.x, lane = tid & 31u, full = 0xffffffffu;
  for (;;) {
    __syncthreads();  // the previous job's shared data is read no more
    if (tid == 0) {
      // a slot beyond its segment's jobs: on to the next segment's first
      uint32_t t;
      int s = 0;
      for (;;) {
        t = atomicAdd(counter, 1u);
        if (t >= total_slots) break;
        int lo = 0, hi = S - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (segs[mid].job_base <= t) lo = mid; else hi = mid - 1;
        }
        s = lo;
        if (segs[s].narrow == (sizeof(T) == 4 ? 1u : 0u) && t - segs[s].job_base < njobs[s]) break;
        if (s + 1 >= S) {
          t = total_slots;
          break;
        }
        atomicMax(counter, segs[s + 1].job_base);
      }
      sm.slot = t;
      sm.seg = s;
      s_cnt[0] = s_cnt[1] = 0;
    }
    __syncthreads();
    const uint32_t slot = sm.slot;
    if (slot >= total_slots) return;
    SortSeg& sg = segs[sm.seg];
    const uint4 job = jobs[slot];
    const bool split = (job.x & kJobSplit) != 0u;
    const uint32_t b = sg.bits, rem = 3 * b - sg.bin_bits, N = job.w;
    const T org = (T)((unsigned long long)(job.x & 0xffffu) << rem);
    const T* src = seg_keys(split ? keys1 : keys0, sg, stride) + job.z;
    T* dst = seg_keys(split ? keys0 : keys1, sg, stride) + job.z;
    uint32_t written = 0, cY = 0, cX = 0;
    T last = 0;  // the greatest key written
    // order the n keys of a, write the distinct ones, count the columns and slabs
    // that they open
    auto emit = [&](T* a, uint32_t n, uint32_t bits) {
      if (n > 1) {
        T* r = bin_block_order<T>(a, a == buf0 ? buf1 : buf0, n, bits, cnt, sm);
        a = r == buf0 ? buf1 : buf0;
        n = bin_block_unique<T>(r, a, n, sm);
      }
      for (uint32_t e = tid; e < n; e += kBinThreads) {
        const T key = a[e], prev = e > 0 ? a[e - 1] : last;
        const bool first = e == 0 && written == 0;
        cY += first || (key >> b) != (prev >> b) ? 1u : 0u;
        cX += (first ? !(job.x & kJobGoesOn)
                     : ((unsigned long long)key >> (2 * b)) != ((unsigned long long)prev >> (2 * b)))
                  ? 1u : 0u;
        dst[written + e] = key;
      }
      if (n > 0) last = a[n - 1];
      written += n;
      __syncthreads();  // the buffers are read no more
    };
    // the keys whose bits from nb up, under `mask`, are `part` (all of them with an
    // empty part): their low nb bits set in a map of the block, which is then in
    // order and free of duplicates; `base` is the key of the map's first place
    auto emit_map = [&](uint32_t nb, T base, uint32_t mask, uint32_t part) {
      uint32_t* map = reinterpret_cast<uint32_t*>(buf0);
      const uint32_t words = nb > 5 ? 1u << (nb - 5) : 1u, low = (1u << nb) - 1u;
      for (uint32_t i = tid; i < words; i += kBinThreads) map[i] = 0;
      if (tid == 0) sm.n = 0;
      __syncthreads();
      for (uint32_t e0 = tid; e0 < N; e0 += 8 * kBinThreads) {
        T v[8];
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) {
          const uint32_t e = e0 + k * kBinThreads;
          v[k] = src[e < N ? e : e0] - org;
        }
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) {
          const uint32_t at = (uint32_t)v[k] & low, bit = 1u << (at & 31u);
          if (mask != full && ((uint32_t)(v[k] >> nb) & mask) != part) continue;
          if (!(((volatile uint32_t*)map)[at >> 5] & bit)) atomicOr(map + (at >> 5), bit);
        }
      }
      __syncthreads();
      const uint32_t per = (words + kBinThreads - 1) / kBinThreads, w0 = tid * per;
      const uint32_t w1 = min(words, w0 + per);
      uint32_t sum = 0, tot, cols = 0;
      for (uint32_t i = w0; i < w1; ++i) {
        sum += __popc(map[i]);
        // a map of several columns (at most 32) has whole words of each (b >= 5)
        if (map[i] && nb > b) cols |= 1u << (i >> (b - 5));
      }
      uint32_t run = block_scan_th<kBinThreads>(sum, tot, sm.scan);
      if (cols) atomicOr(&sm.n, cols);
      T key = 0;
      for (uint32_t i = w0; i < w1; ++i) {
        for (uint32_t m = map[i]; m; m &= m - 1) {
          key = base + 32u * i + (uint32_t)__ffs((int)m) - 1u;
          if (run == 0) buf1[0] = key;
          dst[written + run++] = key;
        }
      }
      if (sum && run == tot) buf1[1] = key;
      __syncthreads();
      if (tot > 0) {
        const T lo = buf1[0];
        if (tid == 0) {
          cY += (nb > b ? __popc(sm.n) : 1) - (written > 0 && (lo >> b) == (last >> b) ? 1 : 0);
          cX += (written == 0 ? !(job.x & kJobGoesOn)
                              : ((unsigned long long)lo >> (2 * b)) != ((unsigned long long)last >> (2 * b)))
                    ? 1u : 0u;
        }
        last = buf1[1];
        written += tot;
      }
      __syncthreads();  // the buffers are read no more
    };
    if (tid == 0) sm.n = sg.fallback;
    __syncthreads();
    // (a row's bits below its own; a map of them takes any number of keys)
    const uint32_t left = rem - min(kBinRowBits, rem - b);
    bool fail = sm.n || N > (left <= kBinMapBits ? map_most : kBinRowMax);
    __syncthreads();
    if (N <= CAP) {
      uint32_t bits = rem;
      while ((1u << (bits - rem)) < job.y) ++bits;
#pragma unroll
      for (int i = 0; i < IT; ++i) {
        const uint32_t e = tid + (uint32_t)kBinThreads * i;
        if (e < N) buf0[e] = src[e] - org;
      }
      __syncthreads();
      emit(buf0, N, bits);
    } else if (!fail) {
      // one row of a split with more keys than the block holds
      const T row = (T)((T)(src[0] - org) >> left) << left;
      if (left <= kBinMapBits) {
        emit_map(left, row, full, 0);
      } else {
        // its keys by their next 12 bits, as many of these parts at a time as fit
        constexpr uint32_t R = 1u << kBinBucketBits, PER = R / kBinThreads;
        uint32_t* pre = cnt + R + 4 + kBinWarps * (R / 32);
        const uint32_t sh = left - kBinBucketBits;
        for (uint32_t r = tid; r < R; r += kBinThreads) pre[r] = 0;
        __syncthreads();
        for (uint32_t e0 = tid; e0 < N; e0 += 8 * kBinThreads) {
          T v[8];
#pragma unroll
          for (uint32_t k = 0; k < 8; ++k) {
            const uint32_t e = e0 + k * kBinThreads;
            v[k] = src[e < N ? e : e0] - org;
          }
#pragma unroll
          for (uint32_t k = 0; k < 8; ++k) {
            if (e0 + k * kBinThreads < N) atomicAdd(pre + ((uint32_t)(v[k] >> sh) & (R - 1)), 1u);
          }
        }
        __syncthreads();
        uint32_t c[PER], sum = 0, tot;
#pragma unroll
        for (uint32_t k = 0; k < PER; ++k) {
          c[k] = pre[tid * PER + k];
          sum += c[k];
        }
        uint32_t run = block_scan_th<kBinThreads>(sum, tot, sm.scan);
#pragma unroll
        for (uint32_t k = 0; k < PER; ++k) {
          pre[tid * PER + k] = run;
          run += c[k];
        }
        if (tid == 0) pre[R] = N;
        __syncthreads();
        int walks = 0;
        for (uint32_t r0 = 0; r0 < R && !fail;) {
          // the most parts [r0, r1) that fit (at least one)
          uint32_t r1 = r0 + 1, hi = R;
          while (r1 < hi) {
            const uint32_t mid = (r1 + hi + 1) >> 1;
            if (pre[mid] - pre[r0] <= CAP) r1 = mid; else hi = mid - 1;
          }
          const uint32_t want = pre[r1] - pre[r0];
          if (want > CAP) {
            emit_map(sh, row + ((T)r0 << sh), R - 1, r0);
          } else if (want > 0) {
            if (tid == 0) sm.n = 0;
            __syncthreads();
            for (uint32_t e0 = 0; e0 < N; e0 += 4 * kBinThreads) {
              T v[4];
#pragma unroll
              for (uint32_t k = 0; k < 4; ++k) {
                const uint32_t e = e0 + k * kBinThreads + tid;
                v[k] = src[e < N ? e : 0u] - org;
              }
#pragma unroll
              for (uint32_t k = 0; k < 4; ++k) {
                const uint32_t r = (uint32_t)(v[k] >> sh) & (R - 1);
                const bool in = e0 + k * kBinThreads + tid < N && r >= r0 && r < r1;
                const uint32_t bal = __ballot_sync(full, in);
                uint32_t at = 0;
                if (lane == 0 && bal) at = atomicAdd(&sm.n, (uint32_t)__popc(bal));
                at = __shfl_sync(full, at, 0);
                if (in) buf0[at + __popc(bal & lanemask_lt())] = v[k];
              }
            }
            __syncthreads();
            emit(buf0, want, left);
          }
          r0 = r1;
          fail = ++walks == kBinWalks && r0 < R && pre[r0] < N;
        }
      }
    }
    if (fail) {
      written = 0;
      if (tid == 0) sg.fallback = 1;
    }
    cY = __reduce_add_sync(full, cY);
    cX = __reduce_add_sync(full, cX);
    if (lane == 0 && cY) {
      atomicAdd(&s_cnt[0], cY);
      atomicAdd(&s_cnt[1], cX);
    }
    __syncthreads();
    if (tid == 0) info[slot] = make_uint4(job.z, written, s_cnt[0], s_cnt[1]);
  }
}

// The CGA arrays of every job: heads of columns and slabs among its distinct keys,
// at the places that the counts of the segment's earlier jobs give (a few thousand
// at most: summed by the block, which is cheaper than another launch).  A job's first
// voxel stays in its second word.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_bin_write(const SortSeg* __restrict__ segs, int S,
                                                        uint4* __restrict__ jobs,
                                                        const uint32_t* __restrict__ njobs,
                                                        const T* __restrict__ keys0,
                                                        const T* __restrict__ keys1,
                                                        const uint4* __restrict__ info,
                                                        uint32_t total_slots, uint32_t stride) {
  __shared__ uint32_t s_w[kWarps][2], s_f[3];
  const uint32_t tid = threadIdx.x, lane = tid & 31u, w = tid >> 5, full = 0xffffffffu;
  const uint32_t ltm = lanemask_lt();
  for (uint32_t slot = blockIdx.x; slot < total_slots; slot += gridDim.x) {
    int lo = 0, hi = S - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (segs[mid].job_base <= slot) lo = mid; else hi = mid - 1;
    }
    const SortSeg& sg = segs[lo];
    if (sg.narrow != (sizeof(T) == 4 ? 1u : 0u) || sg.fallback) continue;
    if (slot - sg.job_base >= njobs[lo]) {
      if (lo + 1 >= S) break;
      continue;
    }
    const uint4 q = info[slot];
    uint32_t fu = 0, fy = 0, fx = 0;
    for (uint32_t j = sg.job_base + tid; j < slot; j += kThreads) {
      const uint4 c = __ldg(info + j);
      fu += c.y;
      fy += c.z;
      fx += c.w;
    }
    __syncthreads();
    if (tid < 3) s_f[tid] = 0;
    __syncthreads();
    fu = __reduce_add_sync(full, fu);
    fy = __reduce_add_sync(full, fy);
    fx = __reduce_add_sync(full, fx);
    if (lane == 0) {
      atomicAdd(&s_f[0], fu);
      atomicAdd(&s_f[1], fy);
      atomicAdd(&s_f[2], fx);
    }
    __syncthreads();
    const uint3 f = make_uint3(s_f[0], s_f[1], s_f[2]);
    const uint32_t jx = jobs[slot].x;
    if (tid == 0) jobs[slot].y = f.x;
    const uint32_t b = sg.bits, rem = 3 * b - sg.bin_bits, m = (1u << b) - 1u;
    const unsigned long long org = (unsigned long long)(jx & 0xffffu) << rem;
    const bool goes_on = (jx & kJobGoesOn) != 0u;
    const Levels& O = sg.out;
    const T* a = seg_keys((jx & kJobSplit) ? keys0 : keys1, sg, stride) + q.x;
    bool bad = false;
    uint32_t rY = f.y, rX = f.z;
    // rounds of four keys a thread: warp w takes 128 consecutive ones
    for (uint32_t e0 = 0; e0 < q.y; e0 += 4 * kThreads) {
      T key[4];
      uint32_t Y[4], X[4], ny = 0, nx = 0;
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) {
        const uint32_t e = e0 + 128 * w + 32 * i + lane;
        const bool v = e < q.y;
        key[i] = v ? __ldg(a + e) : (T)0;
      }
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) {
        const uint32_t e = e0 + 128 * w + 32 * i + lane;
        const bool v = e < q.y;
        T prev = __shfl_up_sync(full, key[i], 1);
        if (lane == 0) prev = v && e > 0 ? __ldg(a + e - 1) : (T)0;
        Y[i] = __ballot_sync(full, v && (e == 0 || (key[i] >> b) != (prev >> b)));
        X[i] = __ballot_sync(full, v && (e == 0 ? !goes_on
                                                : ((unsigned long long)key[i] >> (2 * b)) !=
                                                      ((unsigned long long)prev >> (2 * b))));
        ny += __popc(Y[i]);
        nx += __popc(X[i]);
      }
      __syncthreads();
      if (lane == 0) {
        s_w[w][0] = ny;
        s_w[w][1] = nx;
      }
      __syncthreads();
      uint32_t by = rY, bx = rX;
#pragma unroll
      for (uint32_t x = 0; x < (uint32_t)kWarps; ++x) {
        const uint32_t cy = s_w[x][0], cx = s_w[x][1];
        if (x < w) {
          by += cy;
          bx += cx;
        }
        rY += cy;
        rX += cx;
      }
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) {
        const uint32_t e = e0 + 128 * w + 32 * i + lane;
        const uint32_t pu = f.x + e, py = by + __popc(Y[i] & ltm), px = bx + __popc(X[i] & ltm);
        if (e < q.y) {
          if (pu < O.cap) O.idx0[pu] = (uint16_t)((uint32_t)key[i] & m); else bad = true;
        }
        if ((Y[i] >> lane) & 1u) {
          if (py < O.cap1) {
            O.idx1[py] = (uint16_t)((uint32_t)(key[i] >> b) & m);
            O.ptr1[py] = pu;
          } else {
            bad = true;
          }
        }
        if ((X[i] >> lane) & 1u) {
          if (px < O.cap2) {
            O.idx2[px] = (uint16_t)((org + (unsigned long long)key[i]) >> (2 * b));
            O.ptr2[px] = py;
          } else {
            bad = true;
          }
        }
        by += __popc(Y[i]);
        bx += __popc(X[i]);
      }
    }
    if (bad) atomicOr(&O.hdr->err, kErrInternal);
    if (slot - sg.job_base + 1 == njobs[lo] && tid == 0) {
      // the segment's last job: level sizes and sentinels
      const uint32_t U = f.x + q.y, G = f.y + q.z, H = f.z + q.w;
      if (G <= O.cap1) O.ptr1[G] = U;
      if (H <= O.cap2) O.ptr2[H] = G;
      O.hdr->cnt[0] = U;
      O.hdr->cnt[1] = G;
      O.hdr->cnt[2] = H;
    }
  }
}

// The Value array of the one segment, a job per block: the job's distinct keys and
// their sums in shared memory, every point of the job added to its voxel's.  A table
// of the keys' top bits gives the few keys that a point has to be compared with (a
// bisection of all of them took the kernel from 270 to 526 us, bound by shared-memory
// loads).  The channels' sums have 16 bits each, two to a word, which the count bounds
// (257 * 255 < 2^16); a job with a voxel of more points sums its channels again, two
// at a time in 32 bits.  Up to kBinPacked points the count is the upper half of the
// third channel's word, which no voxel's points can then run over.  A point needs no search of the CGA and no atomic in global
// memory: 15M rows of 3 channels that way took 1010 us for the sums alone.
template <typename T>
constexpr uint32_t bin_values_cap() { return sizeof(T) == 4 ? 6144 : 4096; }  // keys at a time
constexpr uint32_t kBinDirBits = 12;
// the most points n with n counts and n sums of 255 in a word: n * (2^16 + 255) < 2^32
constexpr uint32_t kBinPacked = 0xffffffffu / (65536u + 255u);
template <typename T>
constexpr size_t bin_values_smem() {
  return (sizeof(T) + 12) * (size_t)bin_values_cap<T>() + (sizeof(uint32_t) << kBinDirBits);
}

template <typename T>
__global__ void __launch_bounds__(kBinThreads, 2)
    k_bin_values(const SortSeg* __restrict__ segs, const uint4* __restrict__ jobs,
                 const uint32_t* __restrict__ njobs, const T* __restrict__ keys0,
                 const T* __restrict__ keys1, const uint32_t* __restrict__ rows0,
                 const uint32_t* __restrict__ rows1, const uint4* __restrict__ info,
                 uint32_t stride, ValueInput in, uint8_t* __restrict__ values) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  constexpr uint32_t CAP = bin_values_cap<T>();
  T* s_key = reinterpret_cast<T*>(s_raw);
  uint32_t* s_sum = reinterpret_cast<uint32_t*>(s_key + CAP);  // channels 0, 1
  uint32_t* s_sum2 = s_sum + CAP;                              // channels 2, 3
  uint32_t* s_num = s_sum2 + CAP;
  uint16_t* s_dir = reinterpret_cast<uint16_t*>(s_num + CAP);  // {first, last} key
  const uint32_t tid = threadIdx.x;
  const SortSeg& sg = segs[0];
  if (sg.narrow != (sizeof(T) == 4 ? 1u : 0u) || sg.fallback) return;
  const uint32_t C = in.channels;
  const bool first = in.policy == kValueFirst;
  const uint32_t rem = 3 * sg.bits - sg.bin_bits;
  for (uint32_t slot = blockIdx.x; slot < njobs[0]; slot += gridDim.x) {
    const uint4 job = jobs[slot], q = info[slot];
    const bool split = (job.x & kJobSplit) != 0u;
    const T org = (T)((unsigned long long)(job.x & 0xffffu) << rem);
    const T* src = seg_keys(split ? keys1 : keys0, sg, stride) + job.z;
    const T* key = seg_keys(split ? keys0 : keys1, sg, stride) + q.x;
    const uint32_t* row = (split ? rows1 : rows0) + job.z;
    const uint32_t N = job.w;
    // the count takes the place of a fourth channel where the word holds it
    const bool packed = C <= 3 && N <= kBinPacked;
    for (uint32_t u0 = 0; u0 < q.y; u0 += CAP) {
      const uint32_t n = min(CAP, q.y - u0);
      const T lo = __ldg(key + u0);
      const T span = __ldg(key + u0 + n - 1) - lo;
      uint32_t shift = 0;
      while ((span >> shift) >> kBinDirBits) ++shift;
      __syncthreads();
      for (uint32_t e = tid; e < n; e += kBinThreads) {
        const T k = __ldg(key + u0 + e) - lo;
        const uint32_t d = (uint32_t)(k >> shift);
        s_key[e] = k;
        if (e == 0 || (uint32_t)((T)(__ldg(key + u0 + e - 1) - lo) >> shift) != d) s_dir[2 * d] = (uint16_t)e;
        if (e + 1 == n || (uint32_t)((T)(__ldg(key + u0 + e + 1) - lo) >> shift) != d) {
          s_dir[2 * d + 1] = (uint16_t)e;
        }
        s_sum[e] = first ? 0xffffffffu : 0u;
        s_sum2[e] = s_num[e] = 0;
      }
      __syncthreads();
      // add(voxel, row word) for every point with a voxel among the n
      const T from = org + lo;
      const bool all = n == q.y;
      auto points = [&](auto add) {
        for (uint32_t e0 = tid; e0 < N; e0 += 4 * kBinThreads) {
          T v[4];
          uint32_t r[4];
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t e = e0 + k * kBinThreads < N ? e0 + k * kBinThreads : e0;
            v[k] = __ldg(src + e) - from;
            r[k] = __ldg(row + e);
          }
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k) {
            if (e0 + k * kBinThreads >= N || (!all && v[k] > span)) continue;
            const uint32_t d = reinterpret_cast<const uint32_t*>(s_dir)[(uint32_t)(v[k] >> shift)];
            uint32_t a = d & 0xffffu, b = d >> 16;
            while (b > a + 3) {
              const uint32_t mid = (a + b) >> 1;
              if (s_key[mid] < v[k]) a = mid + 1; else b = mid;
            }
            while (a < b && s_key[a] != v[k]) ++a;
            add(a, r[k]);
          }
        }
      };
      bool many = false;
      if (first) {
        points([&](uint32_t v, uint32_t r) { atomicMin(s_sum + v, r); });
      } else if (packed) {
        points([&](uint32_t v, uint32_t r) {
          atomicAdd(s_sum + v, __byte_perm(r, 0, 0x4140));
          atomicAdd(s_sum2 + v, ((r >> 16) & 0xffu) + 0x10000u);
        });
      } else {
        points([&](uint32_t v, uint32_t r) {
          atomicAdd(s_sum + v, __byte_perm(r, 0, 0x4140));
          if (C > 2) atomicAdd(s_sum2 + v, __byte_perm(r, 0, 0x4342));
          atomicAdd(s_num + v, 1u);
        });
      }
      __syncthreads();
      if (!first) {
        // a sum runs over only where the count is more than 257, and a packed one then
        // adds its carries to the count, which stays below 2^16 (kBinPacked)
        for (uint32_t e = tid; e < n; e += kBinThreads) {
          if (packed) s_num[e] = s_sum2[e] >> 16;
          many |= s_num[e] > 257u;
        }
        many = __syncthreads_or(many);
      }
      uint8_t* out = values + ((size_t)job.y + u0) * C;
      if (first) {
        for (uint32_t e = tid; e < n; e += kBinThreads) {
          const uint8_t* p = in.attr + (size_t)s_sum[e] * C;
          for (uint32_t c = 0; c < C; ++c) out[(size_t)e * C + c] = __ldg(p + c);
        }
      } else if (!many) {
        // round half up by the reciprocal: a quotient that is no whole number is at
        // least 1/257 from the next one, the product within 1/16000 of the quotient
        for (uint32_t e = tid; e < n; e += kBinThreads) {
          const uint32_t k = s_num[e], x = s_sum[e], y = s_sum2[e];
          const float inv = 1.0f / (float)k;
          const uint32_t sum[4] = {x & 0xffffu, x >> 16, y & 0xffffu, y >> 16};
#pragma unroll
          for (uint32_t c = 0; c < 4; ++c) {
            if (c < C) out[(size_t)e * C + c] = (uint8_t)((float)(sum[c] + k / 2) * inv + 0x1p-10f);
          }
        }
      } else {
        if (packed) {  // the counts may have carries in them
          for (uint32_t e = tid; e < n; e += kBinThreads) s_num[e] = 0;
          __syncthreads();
          points([&](uint32_t v, uint32_t) { atomicAdd(s_num + v, 1u); });
        }
        for (uint32_t c = 0; c < C; c += 2) {
          __syncthreads();
          for (uint32_t e = tid; e < n; e += kBinThreads) s_sum[e] = s_sum2[e] = 0;
          __syncthreads();
          points([&](uint32_t v, uint32_t r) {
            atomicAdd(s_sum + v, (r >> (8 * c)) & 0xffu);
            if (c + 1 < C) atomicAdd(s_sum2 + v, (r >> (8 * c + 8)) & 0xffu);
          });
          __syncthreads();
          for (uint32_t e = tid; e < n; e += kBinThreads) {
            const uint32_t k = s_num[e];
            out[(size_t)e * C + c] = (uint8_t)((s_sum[e] + k / 2) / k);
            if (c + 1 < C) out[(size_t)e * C + c + 1] = (uint8_t)((s_sum2[e] + k / 2) / k);
          }
        }
      }
    }
  }
}

}  // namespace

}  // namespace libcga
