// k-means of a CGA's voxels (Sec. V-D) by cells: the same Lloyd passes, with
// whole groups of voxels labelled at once.
//
// A pass of eight exact distances per voxel is bound by integer instructions
// (8.5 warp instructions a voxel and 7% of HBM bandwidth in the per-voxel form,
// k_km_assign).  Most voxels need none of them: for two centres C and L the
// difference d_C(v) - d_L(v) is linear in v, so its minimum over a box is
// exact at a corner, and a group of voxels whose box lies on L's side of every
// bisector takes label L as a whole, its coordinate sums known in advance.
// Only groups that a bisecting plane cuts (about one in twenty on a surface
// scene) look at their voxels, and then only at the centres the box leaves.
//
//   k_kc_count    voxels per cell of a dense grid of at most 128 cells per axis
//   k_kc_scan     cell offsets; cells split into chunks of at most kKcChunk voxels
//   k_kc_scatter  the voxels in cell order, 32 bits each (offsets in the cell)
//   k_kc_stats    box and coordinate sums of every chunk; the box of the cloud
//   k_kc_loop     all passes in one launch, a pass starting when the one before is done
//   k_kc_labels   labels in CGA order from the cells' remaining centres
//
// The chunk bound keeps the work even when a cell holds most of the cloud, and
// lets the coordinate sums of 32 chunks fit 32 bits.  Sums are exact integers
// and a chunk's label is decided exactly, so the result equals the per-voxel
// form whatever the order of the voxels inside a cell.
//
// Measured (GB300, two frames of 19.9M voxels, b = 12, 47 and 44 passes, both
// together): 24.0 ms voxel by voxel (0.25 ms a pass and 8 us for its centres),
// 3.0 ms here when a grid barrier ended each pass and the blocks' sums lay block by
// block: scatter 0.27, count 0.16, labels 0.13, stats 0.11, scan 0.05, the rest the loop
// (24 us a pass: the latency of the mixed chunks' loads and the barrier).  The passes in
// parts, sums word by word: 20M voxels, b = 12, 37 passes 1160 -> 1000 us, b = 10, 64
// passes 1257 -> 945, 1M voxels, 27 passes 562 -> 401.  (With the sums block by block the
// parts took 2% more than the barrier: each block reads 32 words of every block, a
// sector each.)  Chunks of 1024 voxels with all remaining centres measured per
// voxel took 4.6 ms in the loop: too few mixed chunks to share among 4864 warps.
// The voxel-by-voxel form stays for runs of few passes (cells_pay) and for allocators
// without room for the cells.
#include <algorithm>
#include <atomic>

#include "k_walk.cuh"

namespace libcga {

namespace {

constexpr uint32_t kKcChunk = 256;
static_assert((uint64_t)kKcChunk * 32u * 65536u <= (1ull << 31), "sums of a warp's chunks");
constexpr uint32_t kKcScanTile = 2048;   // cells per block of the scan
constexpr int kKcLoopThreads = 1024;
constexpr int kKcPerSm = 6;
constexpr uint32_t kKcNone = 0xFEu;      // chunk state before the first pass
constexpr uint32_t kKcMixed = 0xFFu;     // labels kept voxel by voxel
constexpr uint32_t kKcWords = kKmClusters * 4;  // a block's sums, a warp each
constexpr uint32_t kKcChangedBit = 48;          // of the first count: a label changed

struct KcState {
  uint32_t box[6];   // least y, z (box[1..2]), greatest y, z (box[4..5])
  uint32_t nchunks;
  uint32_t done;     // parts of passes done
  int centre[2][kKmClusters * 3];  // centres of the even and the odd passes' labels
  int used[kKmClusters * 3];       // of the last one's
};

// Cell grid: 2^cb cells of 2^shift voxels per axis.
struct KcGrid {
  uint32_t cb, shift;
};

struct KcView {
  KcState* st;
  uint32_t* cell;     // per cell: count, then cursor, then remaining centres (bit set)
  uint32_t* look;     // scan look-back, 2 words per tile, then the tile counter
  uint32_t* taken;    // per part: passes of it that a block has taken
  uint4* recA;        // chunk: first voxel, count, least, greatest offset in the cell
  uint4* recB;        // chunk: sums of x, y, z; cell
  uint8_t* state;     // chunk: label of all its voxels, kKcMixed or kKcNone
  uint32_t* vox;      // voxels in cell order: x | y << 9 | z << 18 in the cell
  uint8_t* vlab;      // their labels while the chunk is mixed
  unsigned long long* part;  // [2][kKcWords][blocks]
  KcGrid grid;
  uint32_t ncells, max_chunks;
};

size_t align_up(size_t v) { return (v + 255) & ~(size_t)255; }

// Cells per axis: no more than 128, than the grid has voxels, or than give
// about one cell per voxel; cells of at most 512 voxels per axis (9-bit offsets).
KcGrid kc_grid(uint32_t bits, uint64_t cap) {
  uint32_t lg = 0;
  while ((1ull << lg) < cap) ++lg;
  KcGrid g;
  g.cb = std::min<uint32_t>(std::min<uint32_t>(bits, 7u), std::max<uint32_t>((lg + 2) / 3, 2u));
  if (bits > 9u) g.cb = std::max<uint32_t>(g.cb, bits - 9u);
  g.shift = bits - g.cb;
  return g;
}

uint32_t scan_tiles(uint32_t ncells) { return (ncells + kKcScanTile - 1) / kKcScanTile; }

__device__ __forceinline__ uint32_t kc_cell(const KcGrid& g, uint32_t x, uint32_t y, uint32_t z) {
  return ((x >> g.shift) << (2 * g.cb)) | ((y >> g.shift) << g.cb) | (z >> g.shift);
}

__global__ void k_kc_init(KcState* st) {
  const uint32_t t = threadIdx.x;
  if (t < 3) {
    st->box[t] = 0xffffffffu;
    st->box[3 + t] = 0;
  }
  if (t == 0) {
    st->nchunks = 0;
    st->done = 0;
  }
}

// Runs of one cell inside a lane group: `heads` has a bit per lane that opens
// one.  Neighbouring voxels (a column's z run, then the next column's) share
// their cell, so one atomic serves a run.
__device__ __forceinline__ uint32_t run_heads(uint32_t id, uint32_t lane) {
  const uint32_t prev = __shfl_up_sync(0xffffffffu, id, 1);
  return __ballot_sync(0xffffffffu, lane == 0 || id != prev);
}
__device__ __forceinline__ uint32_t run_length(uint32_t heads, uint32_t lane) {
  const uint32_t later = lane == 31 ? 0u : heads >> (lane + 1);
  return later ? (uint32_t)__ffs((int)later) : 32u - lane;
}

__global__ void __launch_bounds__(kThreads, kKcPerSm) k_kc_count(Levels a, KcView v) {
  uint32_t begin, end;
  walk_range((uint32_t)a.hdr->cnt[0], begin, end);
  const uint32_t lane = threadIdx.x & 31u;
  walk_voxels(a, begin, end, [&](uint32_t, uint32_t valid, const uint32_t* x, const uint32_t* y,
                                 const uint32_t* z) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      const bool ok = (valid >> k) & 1u;
      const uint32_t id = ok ? kc_cell(v.grid, x[k], y[k], z[k]) : 0xffffffffu;
      const uint32_t heads = run_heads(id, lane);
      if (ok && ((heads >> lane) & 1u)) atomicAdd(v.cell + id, run_length(heads, lane));
    }
  });
}

// Exclusive scan of the counts (voxels and chunks together): each cell's first
// voxel replaces its count, and its chunks are listed.
__global__ void __launch_bounds__(kThreads) k_kc_scan(KcView v, unsigned int* err) {
  constexpr uint32_t PER = kKcScanTile / kThreads;
  __shared__ unsigned long long s_warp[kWarps];
  __shared__ uint32_t s_tile, s_excl[2];
  const uint32_t tid = threadIdx.x;
  const uint32_t tiles = (v.ncells + kKcScanTile - 1) / kKcScanTile;
  if (tid == 0) s_tile = atomicAdd(v.look + 2 * tiles, 1u);
  __syncthreads();
  const uint32_t t = s_tile, c0 = t * kKcScanTile + tid * PER;
  uint32_t n[PER];
  unsigned long long sum = 0;
#pragma unroll
  for (uint32_t i = 0; i < PER; i += 4) {
    const uint4 q = *reinterpret_cast<const uint4*>(v.cell + c0 + i);
    n[i] = q.x;
    n[i + 1] = q.y;
    n[i + 2] = q.z;
    n[i + 3] = q.w;
  }
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    sum += (unsigned long long)n[i] |
           ((unsigned long long)((n[i] + kKcChunk - 1) / kKcChunk) << 32);
  }
  unsigned long long tot = 0;
  const unsigned long long ex = block_excl_scan(sum, tot, s_warp);
  if (tid < 2) {
    const uint32_t run = (uint32_t)(tot >> (32 * tid));
    uint32_t* my = v.look + 2 * t + tid;
    uint32_t excl = 0;
    st_relaxed(my, (t == 0 ? kFlagInc : kFlagAgg) | run);
    if (t > 0) {
      excl = lookback(v.look + tid, 2, t, 0, err);
      st_relaxed(my, kFlagInc | ((excl + run) & kValMask));
    }
    s_excl[tid] = excl;
    if (tid == 1 && t + 1 == tiles) v.st->nchunks = min(excl + run, v.max_chunks);
  }
  __syncthreads();
  uint32_t start = s_excl[0] + (uint32_t)ex, j = s_excl[1] + (uint32_t)(ex >> 32);
#pragma unroll
  for (uint32_t i = 0; i < PER; ++i) {
    for (uint32_t q = 0; q < n[i]; q += kKcChunk) {
      if (j < v.max_chunks) {
        v.recA[j] = make_uint4(start + q, min(kKcChunk, n[i] - q), 0u, 0u);
        v.recB[j].w = c0 + i;
      }
      ++j;
    }
    const uint32_t first = start;
    start += n[i];
    n[i] = first;
  }
#pragma unroll
  for (uint32_t i = 0; i < PER; i += 4) {
    *reinterpret_cast<uint4*>(v.cell + c0 + i) = make_uint4(n[i], n[i + 1], n[i + 2], n[i + 3]);
  }
}

__global__ void __launch_bounds__(kThreads, kKcPerSm) k_kc_scatter(Levels a, KcView v) {
  const uint32_t u = (uint32_t)a.hdr->cnt[0];
  uint32_t begin, end;
  walk_range(u, begin, end);
  const uint32_t lane = threadIdx.x & 31u, m = (1u << v.grid.shift) - 1u;
  const uint32_t le = 0xffffffffu >> (31u - lane);
  walk_voxels(a, begin, end, [&](uint32_t, uint32_t valid, const uint32_t* x, const uint32_t* y,
                                 const uint32_t* z) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      const bool ok = (valid >> k) & 1u;
      const uint32_t id = ok ? kc_cell(v.grid, x[k], y[k], z[k]) : 0xffffffffu;
      const uint32_t heads = run_heads(id, lane);
      uint32_t base = 0;
      if (ok && ((heads >> lane) & 1u)) base = atomicAdd(v.cell + id, run_length(heads, lane));
      const uint32_t head = 31u - (uint32_t)__clz((int)(heads & le));
      const uint32_t pos = __shfl_sync(0xffffffffu, base, head) + (lane - head);
      if (ok && pos < u) v.vox[pos] = (x[k] & m) | (y[k] & m) << 9 | (z[k] & m) << 18;
    }
  });
}

// Box and sums of every chunk (a warp each), the box of the whole cloud, and
// the cells' masks cleared for k_kc_loop's last step.
__global__ void __launch_bounds__(kThreads) k_kc_stats(KcView v) {
  __shared__ uint32_t s_box[4];  // least y, z; greatest y, z
  const uint32_t full = 0xffffffffu, lane = threadIdx.x & 31u;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t n = v.st->nchunks, cb = v.grid.cb, sh = v.grid.shift, cm = (1u << cb) - 1u;
  if (threadIdx.x < 4) s_box[threadIdx.x] = threadIdx.x < 2 ? full : 0u;
  __syncthreads();
  uint32_t by0 = full, bz0 = full, by1 = 0, bz1 = 0;
  for (uint32_t j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < n; j += warps) {
    const uint4 A = v.recA[j];
    const uint32_t id = v.recB[j].w;
    uint32_t lo[3] = {full, full, full}, hi[3] = {0, 0, 0}, sum[3] = {0, 0, 0};
    for (uint32_t i = lane; i < A.y; i += 32) {
      const uint32_t w = __ldg(v.vox + A.x + i);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const uint32_t c = (w >> (9 * a)) & 511u;
        lo[a] = min(lo[a], c);
        hi[a] = max(hi[a], c);
        sum[a] += c;
      }
    }
    const uint32_t o[3] = {(id >> (2 * cb)) << sh, ((id >> cb) & cm) << sh, (id & cm) << sh};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lo[a] = __reduce_min_sync(full, lo[a]);
      hi[a] = __reduce_max_sync(full, hi[a]);
      sum[a] = __reduce_add_sync(full, sum[a]) + A.y * o[a];
    }
    by0 = min(by0, o[1] + lo[1]);
    by1 = max(by1, o[1] + hi[1]);
    bz0 = min(bz0, o[2] + lo[2]);
    bz1 = max(bz1, o[2] + hi[2]);
    if (lane == 0) {
      v.recA[j] = make_uint4(A.x, A.y, lo[0] | lo[1] << 9 | lo[2] << 18,
                             hi[0] | hi[1] << 9 | hi[2] << 18);
      v.recB[j] = make_uint4(sum[0], sum[1], sum[2], id);
      v.state[j] = (uint8_t)kKcNone;
      v.cell[id] = 0;
    }
  }
  if (lane == 0) {
    atomicMin(&s_box[0], by0);
    atomicMin(&s_box[1], bz0);
    atomicMax(&s_box[2], by1);
    atomicMax(&s_box[3], bz1);
  }
  __syncthreads();
  if (threadIdx.x < 2) atomicMin(&v.st->box[1 + threadIdx.x], s_box[threadIdx.x]);
  else if (threadIdx.x < 4) atomicMax(&v.st->box[2 + threadIdx.x], s_box[threadIdx.x]);
}

// Nearest of the centres in `mask` (at least one) to voxel (x, y, z): the least
// exact squared distance in 1/256 voxel, the lower cluster on a tie.
__device__ __forceinline__ uint32_t nearest(const int* c, uint32_t mask, uint32_t x, uint32_t y,
                                            uint32_t z) {
  const int vx = (int)(x << 8), vy = (int)(y << 8), vz = (int)(z << 8);
  unsigned long long bd = ~0ull;
  uint32_t best = 0;
  for (uint32_t m = mask; m != 0u; m &= m - 1u) {
    const uint32_t k = (uint32_t)__ffs((int)m) - 1u;
    const int dx = vx - c[3 * k], dy = vy - c[3 * k + 1], dz = vz - c[3 * k + 2];
    const unsigned long long d = (unsigned long long)((long long)dx * dx) +
                                 (unsigned long long)((long long)dy * dy) +
                                 (unsigned long long)((long long)dz * dz);
    if (d < bd) {
      bd = d;
      best = k;
    }
  }
  return best;
}

// The centres that can be the nearest of some voxel of the box [lo, hi]
// (voxels): L, the nearest to its middle, and every C whose d_C - d_L is not
// positive (not even zero when C comes after L) over the whole box.
__device__ __forceinline__ uint32_t box_centres(const int* c, const long long* q, const int* lo,
                                                const int* hi) {
  uint32_t L = 0;
  long long bd = 0x7fffffffffffffffll;
#pragma unroll
  for (uint32_t k = 0; k < kKmClusters; ++k) {
    long long d = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int e = (lo[a] + hi[a]) * 128 - c[3 * k + a];
      d += (long long)e * e;
    }
    if (d < bd) {
      bd = d;
      L = k;
    }
  }
  uint32_t mask = 1u << L;
  const long long qL = q[L];
  const int l0 = c[3 * L], l1 = c[3 * L + 1], l2 = c[3 * L + 2];
#pragma unroll
  for (uint32_t k = 0; k < kKmClusters; ++k) {
    const int d0 = c[3 * k] - l0, d1 = c[3 * k + 1] - l1, d2 = c[3 * k + 2] - l2;
    // the greatest v . (C - L) over the box, voxels
    const long long m = (long long)d0 * (d0 > 0 ? hi[0] : lo[0]) +
                        (long long)d1 * (d1 > 0 ? hi[1] : lo[1]) +
                        (long long)d2 * (d2 > 0 ? hi[2] : lo[2]);
    const long long least = q[k] - qL - 512 * m;
    if (k != L && (least < 0 || (least == 0 && k < L))) mask |= 1u << k;
  }
  return mask;
}

// A pass is as many parts as the launch has blocks; its chunks are dealt out over them,
// and block i takes part i of every pass, whose voxels it then finds in its L1.  The
// blocks need not all be resident: one that waits longer than kKcHelpNs for a pass takes
// over a part that no block has begun.  (Parts taken in order by whichever block comes
// first: no slower where few chunks are mixed, but 40 passes over 20M uniform voxels, most
// of them mixed, 3.8 ms against 3.1.)  A part taken keeps its pass from ending, so the sums
// and centres of the pass before stay until the part is done.  Every part sums the pass
// before for itself and moves that pass's centres.  In place of the pass after the last
// one each block leaves its part of the results.
constexpr unsigned long long kKcHelpNs = 30000;

// Waits until `target` parts are done (0), or a part of `pass` that no block has begun is
// taken over (1, its number in `part`), or the wait gives up (2).
__device__ __forceinline__ uint32_t wait_pass(const KcView& v, uint32_t parts, uint32_t pass,
                                              uint32_t target, unsigned int* err,
                                              uint32_t* s_word, uint32_t& part) {
  if (threadIdx.x < 32) {
    const uint32_t full = 0xffffffffu, lane = threadIdx.x;
    const unsigned long long t0 = global_ns();
    uint32_t r = 0, at = 0, spins = 0;
    for (;;) {
      uint32_t seen = 0;
      if (lane == 0) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];"
                     : "=r"(seen) : "l"(&v.st->done) : "memory");
      }
      if (__shfl_sync(full, seen, 0) >= target) break;
      if ((++spins & 15u) != 0) continue;
      const unsigned long long dt = __shfl_sync(full, global_ns() - t0, 0);
      if (dt > kWaitLimitNs) {
        if (lane == 0) atomicOr(err, kErrTimeout);
        r = 2;
        break;
      }
      for (uint32_t p0 = 0; dt > kKcHelpNs && r == 0 && p0 < parts; p0 += 32) {
        const uint32_t p = p0 + lane;
        uint32_t todo = __ballot_sync(full, p < parts && __ldcg(v.taken + p) == pass);
        for (; todo && r == 0; todo &= todo - 1) {
          at = p0 + (uint32_t)__ffs((int)todo) - 1u;
          if (lane == 0) r = atomicCAS(v.taken + at, pass, pass + 1) == pass ? 1u : 0u;
          r = __shfl_sync(full, r, 0);
        }
      }
      if (r != 0) break;
    }
    if (lane == 0) *s_word = r | at << 2;
  }
  __syncthreads();
  const uint32_t word = *s_word;
  __syncthreads();  // (the word is read no more)
  part = word >> 2;
  return word & 3u;
}

__global__ void __launch_bounds__(kKcLoopThreads, 1)
    k_kc_loop(Levels a, KcView v, uint32_t max_iter, long long* centres,
              unsigned long long* counts, uint32_t* iters) {
  constexpr uint32_t W = kKcLoopThreads / 32;
  static_assert(W == kKcWords, "a warp per word of the sums");
  __shared__ int s_c[kKmClusters * 3];
  __shared__ long long s_q[kKmClusters];
  __shared__ unsigned long long s_part[W][kKmClusters * 4 + 1];
  __shared__ unsigned long long s_tot[kKcWords + 1];  // the sums; parts with a change
  __shared__ uint32_t s_own, s_word;
  const uint32_t full = 0xffffffffu, tid = threadIdx.x, lane = tid & 31u, w = tid >> 5;
  const uint32_t u = (uint32_t)a.hdr->cnt[0], h = (uint32_t)a.hdr->cnt[2];
  if (u == 0) {
    if (blockIdx.x == 0) {
      if (tid < kKmClusters * 3) centres[tid] = 0;
      if (tid < kKmClusters) counts[tid] = 0;
      if (tid == 0) *iters = 0;
    }
    return;
  }
  const uint32_t nch = v.st->nchunks, cb = v.grid.cb, sh = v.grid.shift, cm = (1u << cb) - 1u;
  const uint32_t parts = gridDim.x, warps = parts * W;
  // the pass in work (a block may start late), and whether this block has its part of it
  uint32_t pass = 0, ready = 0xffffffffu;  // ready: the pass whose centres s_c holds
  if (tid == 0) {
    uint32_t seen;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&v.st->done) : "memory");
    s_word = seen / parts;
    s_own = atomicCAS(v.taken + blockIdx.x, s_word, s_word + 1) == s_word;
  }
  __syncthreads();
  pass = s_word;
  __syncthreads();
  // The chunks of warp gw of a pass: their sums and whether a label changed.  (Written out
  // for the block's own part, whose number is known to be the same for all lanes, and for
  // others: by a number from shared memory the mixed chunks of 20M uniform voxels took a
  // third longer.)
  unsigned long long acc;  // lane l: entry l = label * 4 + {x, y, z sum, count}
  bool changed;
  auto chunks = [&](uint32_t gw) {
    acc = 0;
    changed = false;
    // chunk i of a round goes to lane i / warps of warp i % warps: the mixed
    // chunks, neighbours in the cell order, spread over the warps
    for (uint32_t r = 0; r < nch; r += 32u * warps) {
      const uint32_t j = r + lane * warps + gw;
      const bool ok = j < nch;
      uint4 A = make_uint4(0, 0, 0, 0), B = A;
      uint32_t mask = 0, old = kKcNone;
      if (ok) {
        A = __ldg(v.recA + j);
        B = __ldg(v.recB + j);
        old = v.state[j];
        const int o[3] = {(int)((B.w >> (2 * cb)) << sh), (int)(((B.w >> cb) & cm) << sh),
                          (int)((B.w & cm) << sh)};
        int lo[3], hi[3];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
          lo[ax] = o[ax] + (int)((A.z >> (9 * ax)) & 511u);
          hi[ax] = o[ax] + (int)((A.w >> (9 * ax)) & 511u);
        }
        mask = box_centres(s_c, s_q, lo, hi);
      }
      const bool whole = ok && (mask & (mask - 1u)) == 0u;
      const uint32_t L = whole ? (uint32_t)__ffs((int)mask) - 1u : 0u;
      // whole chunks: label by label
      uint32_t todo = __ballot_sync(full, whole);
      while (todo) {
        const uint32_t l = __shfl_sync(full, L, __ffs((int)todo) - 1);
        const bool mine = whole && L == l;
        todo &= ~__ballot_sync(full, mine);
        const uint32_t sx = __reduce_add_sync(full, mine ? B.x : 0u);
        const uint32_t sy = __reduce_add_sync(full, mine ? B.y : 0u);
        const uint32_t sz = __reduce_add_sync(full, mine ? B.z : 0u);
        const uint32_t sn = __reduce_add_sync(full, mine ? A.y : 0u);
        if ((lane >> 2) == l) {
          const uint32_t e = lane & 3u;
          acc += e == 0 ? sx : (e == 1 ? sy : (e == 2 ? sz : sn));
        }
      }
      if (whole) {
        if (old != kKcMixed) {
          changed = changed || old != L;
        }
        v.state[j] = (uint8_t)L;
      } else if (ok) {
        v.state[j] = (uint8_t)kKcMixed;
      }
      // chunks that were mixed and are whole now: did every voxel have the label?
      uint32_t back = __ballot_sync(full, whole && old == kKcMixed);
      while (back) {
        const uint32_t src = (uint32_t)__ffs((int)back) - 1u;
        back &= back - 1u;
        const uint32_t s0 = __shfl_sync(full, A.x, src), n = __shfl_sync(full, A.y, src);
        const uint32_t l = __shfl_sync(full, L, src);
        for (uint32_t i = lane; i < n; i += 32) changed = changed || v.vlab[s0 + i] != l;
      }
      // mixed chunks, the whole warp on each
      uint32_t mixed = __ballot_sync(full, ok && !whole);
      while (mixed) {
        const uint32_t src = (uint32_t)__ffs((int)mixed) - 1u;
        mixed &= mixed - 1u;
        const uint32_t s0 = __shfl_sync(full, A.x, src), n = __shfl_sync(full, A.y, src);
        const uint32_t id = __shfl_sync(full, B.w, src), mk = __shfl_sync(full, mask, src);
        const uint32_t was = __shfl_sync(full, old, src);
        const uint32_t ox = (id >> (2 * cb)) << sh, oy = ((id >> cb) & cm) << sh,
                       oz = (id & cm) << sh;
        const uint32_t l0 = (uint32_t)__ffs((int)mk) - 1u, rest = mk & (mk - 1u);
        if ((rest & (rest - 1u)) == 0u) {
          // two centres left: the sign of d_l1 - d_l0, linear in the voxel's
          // offset from the cell, l0 on a tie; l1's sums lane by lane, l0's as
          // the chunk's less l1's
          const uint32_t l1 = (uint32_t)__ffs((int)rest) - 1u;
          const int d0 = s_c[3 * l1] - s_c[3 * l0], d1 = s_c[3 * l1 + 1] - s_c[3 * l0 + 1],
                    d2 = s_c[3 * l1 + 2] - s_c[3 * l0 + 2];
          const long long at0 = (long long)d0 * (int)ox + (long long)d1 * (int)oy +
                                (long long)d2 * (int)oz;
          // l1 when 512 (v . d) > q[l1] - q[l0], v . d a whole number
          const long long lim = ((s_q[l1] - s_q[l0]) >> 9) - at0;
          uint32_t sx = 0, sy = 0, sz = 0, sn = 0;
          for (uint32_t i0 = lane; i0 < n; i0 += 128) {
            uint32_t q[4], before[4];
#pragma unroll
            for (uint32_t e = 0; e < 4; ++e) {
              const uint32_t i = i0 + 32 * e;
              q[e] = i < n ? __ldg(v.vox + s0 + i) : 0u;
              before[e] = was != kKcMixed ? was : (i < n ? (uint32_t)v.vlab[s0 + i] : 0u);
            }
#pragma unroll
            for (uint32_t e = 0; e < 4; ++e) {
              const uint32_t i = i0 + 32 * e;
              if (i >= n) break;
              const uint32_t x = q[e] & 511u, y = (q[e] >> 9) & 511u, z = (q[e] >> 18) & 511u;
              const long long t = (long long)d0 * (int)x + (long long)d1 * (int)y +
                                  (long long)d2 * (int)z;
              const bool one = t > lim;
              if (one) {
                sx += x;
                sy += y;
                sz += z;
                ++sn;
              }
              const uint32_t best = one ? l1 : l0;
              changed = changed || before[e] != best;
              if (before[e] != best || was != kKcMixed) v.vlab[s0 + i] = (uint8_t)best;
            }
          }
          sn = __reduce_add_sync(full, sn);
          sx = __reduce_add_sync(full, sx) + sn * ox;
          sy = __reduce_add_sync(full, sy) + sn * oy;
          sz = __reduce_add_sync(full, sz) + sn * oz;
          const uint32_t tx = __shfl_sync(full, B.x, src), ty = __shfl_sync(full, B.y, src),
                         tz = __shfl_sync(full, B.z, src);
          const uint32_t e = lane & 3u;
          const uint32_t v1 = e == 0 ? sx : (e == 1 ? sy : (e == 2 ? sz : sn));
          const uint32_t vt = e == 0 ? tx : (e == 1 ? ty : (e == 2 ? tz : n));
          if ((lane >> 2) == l1) acc += v1;
          if ((lane >> 2) == l0) acc += vt - v1;
          continue;
        }
        for (uint32_t i0 = 0; i0 < n; i0 += 32) {
          const uint32_t i = i0 + lane;
          const bool in = i < n;
          uint32_t x = 0, y = 0, z = 0, best = 0xffu;
          if (in) {
            const uint32_t q = __ldg(v.vox + s0 + i);
            x = ox + (q & 511u);
            y = oy + ((q >> 9) & 511u);
            z = oz + ((q >> 18) & 511u);
            best = nearest(s_c, mk, x, y, z);
            const uint32_t before = was == kKcMixed ? (uint32_t)v.vlab[s0 + i] : was;
            changed = changed || before != best;
            if (before != best || was != kKcMixed) v.vlab[s0 + i] = (uint8_t)best;
          }
          for (uint32_t m = mk; m != 0u; m &= m - 1u) {
            const uint32_t l = (uint32_t)__ffs((int)m) - 1u;
            const bool mine = best == l;
            const uint32_t sn = (uint32_t)__popc(__ballot_sync(full, mine));
            if (sn == 0) continue;
            const uint32_t sx = __reduce_add_sync(full, mine ? x : 0u);
            const uint32_t sy = __reduce_add_sync(full, mine ? y : 0u);
            const uint32_t sz = __reduce_add_sync(full, mine ? z : 0u);
            if ((lane >> 2) == l) {
              const uint32_t e = lane & 3u;
              acc += e == 0 ? sx : (e == 1 ? sy : (e == 2 ? sz : sn));
            }
          }
        }
      }
    }
  };
  bool own = s_own != 0, asked = false;  // asked: for its part of the next pass
  for (;;) {
    uint32_t part = blockIdx.x;
    if (!own) {
      // on to the next pass once this one is done
      const uint32_t r = wait_pass(v, parts, pass, (pass + 1) * parts, &a.hdr->err, &s_word, part);
      if (r == 2) return;
      if (r == 0) {
        ++pass;
        if (!asked && tid == 0) s_own = atomicCAS(v.taken + blockIdx.x, pass, pass + 1) == pass;
        asked = false;
        __syncthreads();
        own = s_own != 0;
        if (!own) continue;
        part = blockIdx.x;
      }
    }
    own = false;
    const uint32_t gw = part * W + w;
    if (ready != pass) {
      bool converged = false;
      if (pass == 0) {
        // corner c of the box: the greatest coordinate of axis ax where bit ax of c is set
        if (tid < kKmClusters * 3) {
          const uint32_t c = tid / 3, ax = tid % 3;
          const uint32_t lo = ax == 0 ? (uint32_t)__ldg(a.idx2) : v.st->box[ax];
          const uint32_t hi = ax == 0 ? (uint32_t)__ldg(a.idx2 + h - 1) : v.st->box[3 + ax];
          s_c[tid] = (int)(256u * (((c >> ax) & 1u) ? hi : lo));
        }
      } else {
        const uint32_t odd = (pass - 1) & 1u;
        const unsigned long long* sums = v.part + (size_t)odd * parts * kKcWords;
        if (tid < kKmClusters * 3) s_c[tid] = __ldcg(&v.st->centre[odd][tid]);
        {
          unsigned long long s = 0;
          for (uint32_t b = lane; b < parts; b += 32) s += __ldcg(sums + w * parts + b);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(full, s, o);
          if (lane == 0) {
            s_tot[w] = s & ((1ull << kKcChangedBit) - 1);
            if (w == 3) s_tot[kKcWords] = s >> kKcChangedBit;
          }
        }
        __syncthreads();
        converged = pass > 1 && s_tot[kKcWords] == 0;
      }
      const bool stop = pass > 0 && (converged || pass >= max_iter);
      if (pass > 0 && !stop && tid < kKmClusters * 3) {
        const unsigned long long n = s_tot[4 * (tid / 3) + 3];
        if (n > 0) s_c[tid] = (int)((256ull * s_tot[4 * (tid / 3) + tid % 3] + n / 2) / n);
      }
      __syncthreads();
      if (tid < kKmClusters) {
        long long q = 0;
        for (int ax = 0; ax < 3; ++ax) q += (long long)s_c[3 * tid + ax] * s_c[3 * tid + ax];
        s_q[tid] = q;
      }
      __syncthreads();
      if (stop) {
        if (part == 0) {
          if (tid < kKmClusters * 3) {
            const int c = s_c[tid];
            const unsigned long long n = s_tot[4 * (tid / 3) + 3];
            v.st->used[tid] = c;
            centres[tid] = converged || n == 0
                               ? c : (int)((256ull * s_tot[4 * (tid / 3) + tid % 3] + n / 2) / n);
          }
          if (tid < kKmClusters) counts[tid] = s_tot[4 * tid + 3];
          if (tid == 0) *iters = pass;
        }
        // the cells' remaining centres, for the labels in CGA order
        for (uint32_t j = gw * 32u + lane; j < nch; j += 32u * warps) {
          const uint4 A = __ldg(v.recA + j);
          const uint32_t id = __ldg(&v.recB[j].w);
          const int o[3] = {(int)((id >> (2 * cb)) << sh), (int)(((id >> cb) & cm) << sh),
                            (int)((id & cm) << sh)};
          int lo[3], hi[3];
#pragma unroll
          for (int ax = 0; ax < 3; ++ax) {
            lo[ax] = o[ax] + (int)((A.z >> (9 * ax)) & 511u);
            hi[ax] = o[ax] + (int)((A.w >> (9 * ax)) & 511u);
          }
          atomicOr(v.cell + id, box_centres(s_c, s_q, lo, hi));
        }
        return;
      }
      ready = pass;
    }
    if (part == 0 && tid < kKmClusters * 3) v.st->centre[pass & 1u][tid] = s_c[tid];
    if (part == blockIdx.x) {
      chunks(blockIdx.x * W + w);
    } else {
      chunks(gw);
    }
    // (the block's part of the next pass, asked for while its last warps work)
    if (part == blockIdx.x) {
      if (tid == 0) s_own = atomicCAS(v.taken + part, pass + 1, pass + 2) == pass + 1;
      asked = true;
    }
    // block sums: entry e of every warp, then one word per entry and block
    s_part[w][lane] = acc;
    const bool any = __syncthreads_or(changed);
    {
      unsigned long long* sums = v.part + (size_t)(pass & 1u) * parts * kKcWords + part;
      unsigned long long s = lane < W ? s_part[lane][w] : 0ull;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(full, s, o);
      if (lane == 0) sums[w * parts] = s | (w == 3 && any ? 1ull << kKcChangedBit : 0ull);
    }
    count_done(&v.st->done);
  }
}

__global__ void __launch_bounds__(kThreads, kKcPerSm)
    k_kc_labels(Levels a, KcView v, uint8_t* __restrict__ labels) {
  __shared__ int s_c[kKmClusters * 3];
  if (threadIdx.x < kKmClusters * 3) s_c[threadIdx.x] = v.st->used[threadIdx.x];
  __syncthreads();
  uint32_t begin, end;
  walk_range((uint32_t)a.hdr->cnt[0], begin, end);
  const uint32_t lane = threadIdx.x & 31u;
  walk_voxels(a, begin, end, [&](uint32_t p, uint32_t valid, const uint32_t* x, const uint32_t* y,
                                 const uint32_t* z) {
    uint32_t m[4];
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      m[k] = ((valid >> k) & 1u) ? __ldg(v.cell + kc_cell(v.grid, x[k], y[k], z[k])) : 0u;
    }
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      if (m[k] == 0u) continue;
      const uint32_t l = (m[k] & (m[k] - 1u)) ? nearest(s_c, m[k], x[k], y[k], z[k])
                                              : (uint32_t)__ffs((int)m[k]) - 1u;
      labels[p + 32 * k + lane] = (uint8_t)l;
    }
  });
}

// Blocks of the loop kernel: one per SM that can hold one (0: none can).
uint32_t loop_blocks() {
  static std::atomic<int> cache{-1};
  int n = cache.load(std::memory_order_relaxed);
  if (n < 0) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_kc_loop, kKcLoopThreads, 0) !=
        cudaSuccess) {
      cudaGetLastError();
      occ = 0;
    }
    n = occ > 0 ? device_sm_count() : 0;
    cache.store(n, std::memory_order_relaxed);
  }
  return (uint32_t)n;
}

size_t kc_layout(uint32_t bits, uint64_t cap, char* base, KcView* out) {
  KcView v{};
  v.grid = kc_grid(bits, cap);
  v.ncells = 1u << (3 * v.grid.cb);
  v.max_chunks = (uint32_t)(std::min<uint64_t>(v.ncells, cap) + cap / kKcChunk + 1);
  const uint32_t tiles = scan_tiles(v.ncells);
  size_t p = 0;
  auto take = [&](size_t bytes) {
    char* r = base + p;
    p += align_up(bytes);
    return r;
  };
  v.st = reinterpret_cast<KcState*>(take(sizeof(KcState)));
  v.look = reinterpret_cast<uint32_t*>(take((2 * (size_t)tiles + 1) * 4));
  v.taken = reinterpret_cast<uint32_t*>(take(std::max<uint32_t>(loop_blocks(), 1u) * 4));
  v.cell = reinterpret_cast<uint32_t*>(take((size_t)tiles * kKcScanTile * 4));
  v.recA = reinterpret_cast<uint4*>(take((size_t)v.max_chunks * 16));
  v.recB = reinterpret_cast<uint4*>(take((size_t)v.max_chunks * 16));
  v.state = reinterpret_cast<uint8_t*>(take(v.max_chunks));
  v.vox = reinterpret_cast<uint32_t*>(take(cap * 4));
  v.vlab = reinterpret_cast<uint8_t*>(take(cap));
  v.part = reinterpret_cast<unsigned long long*>(
      take(2 * (size_t)std::max<uint32_t>(loop_blocks(), 1u) * kKcWords * 8));
  if (out != nullptr) *out = v;
  return p;
}

}  // namespace

// The cells pay once their tables have cost less than the passes save (of at most
// max_iter passes; the voxel-by-voxel form queues a launch pair for each of those).  In
// us, from runs of 1 to 16 passes over 100 to 20M surface voxels, b = 10, 12 and 16:
// the tables about 35, 14 for each 2^20 cells and 10 for each 2^20 voxels more than what
// the other form starts with; a pass saves 8 (launches), up to 16 more from 8192 voxels
// on and 8 for each 2^20.  Voxel by voxel and by cells: 1000 voxels, b = 16, 1 pass 52
// and 121, 6 passes 144 and 152, 8 passes 182 and 167; 10k, b = 10, 1 pass 63 and 71, 2
// passes 93 and 84; 20M, b = 12, 1 pass 255 and 330, 2 passes 442 and 352.
static bool cells_pay(const KcGrid& g, uint64_t cap, uint32_t max_iter) {
  const double m = (double)cap / (1 << 20);
  const double tables = 35.0 + 14.0 * (double)(1u << (3 * g.cb)) / (1 << 20) + 10.0 * m;
  const double pass = 8.0 + 16.0 * (double)std::min<uint64_t>(cap, 8192) / 8192 + 8.0 * m;
  return pass * max_iter > tables;
}

size_t kmeans_cells_bytes(uint32_t bits, uint64_t cap, uint32_t max_iter) {
  if (cap == 0 || loop_blocks() == 0 || !cells_pay(kc_grid(bits, cap), cap, max_iter)) return 0;
  return kc_layout(bits, cap, nullptr, nullptr);
}

cudaError_t run_kmeans_cells(const Levels& a, uint32_t max_iter, void* scratch, uint8_t* labels,
                             long long* centres, unsigned long long* counts, uint32_t* iters,
                             cudaStream_t stream) {
  KcView v;
  kc_layout(a.bits, a.cap, static_cast<char*>(scratch), &v);
  const uint32_t tiles = scan_tiles(v.ncells);
  // the look-back words, the parts' and the cell counts lie side by side
  cudaError_t e = cudaMemsetAsync(
      v.look, 0, (size_t)(reinterpret_cast<char*>(v.recA) - reinterpret_cast<char*>(v.look)), stream);
  if (e != cudaSuccess) return e;
  k_kc_init<<<1, 32, 0, stream>>>(v.st);
  k_kc_count<<<walk_blocks(a.cap, kKcPerSm), kThreads, 0, stream>>>(a, v);
  k_kc_scan<<<tiles, kThreads, 0, stream>>>(v, &a.hdr->err);
  k_kc_scatter<<<walk_blocks(a.cap, kKcPerSm), kThreads, 0, stream>>>(a, v);
  const unsigned sb = (unsigned)std::min<uint64_t>(((uint64_t)v.max_chunks + 7) / 8,
                                                   (uint64_t)device_sm_count() * 8);
  k_kc_stats<<<sb, kThreads, 0, stream>>>(v);
  k_kc_loop<<<loop_blocks(), kKcLoopThreads, 0, stream>>>(a, v, max_iter, centres, counts, iters);
  k_kc_labels<<<walk_blocks(a.cap, kKcPerSm), kThreads, 0, stream>>>(a, v, labels);
  count_launch(7);
  return cudaGetLastError();
}

}  // namespace libcga
