// The X -> Y -> Z walk of Sec. V-A over a run of consecutive CGA positions, by
// one warp without shared memory or barriers.
//
// A position's column is the number of Y_pointer entries at or below it, so a
// warp that holds the column of the position before its group of 32 needs only
// the starts of the columns that follow: each start inside the group sets one
// bit of a 32-bit mask, and a lane's column is the held one plus the set bits
// at or below its lane.  Every column holds at least one voxel, so 128
// consecutive starts always cover the next 128 positions: they and the 128 z
// entries are eight coalesced loads in flight at once, followed by the gather
// of y.  x changes rarely on coarse grids: one slab that opens inside the group is
// applied by all lanes together.  Where more do, the next 32 are loaded at once, a lane
// each, and applied one after the other.  (Loaded one by one they took a decode of 3M
// LiDAR points at b = 16, whose slabs hold a few tens of voxels, 42 us, by tiles 35; 26
// so.  Without the step for a single slab 20M surface voxels take 65 us, not 61.)
//
// What it replaced: a block of 256 threads expanding a tile of 4096 positions
// through shared memory (scatter of the starts, block max-scans), preceded by
// four dependent warp searches per tile.  The search now runs once per warp
// for its whole run of positions.  Measured on the 20M-voxel surface world:
// decode 127 -> 65 us (240 MB written: 3.7 TB/s), the bits of one projection
// plane 166 -> 110 us, the tree keys 360 -> 264 us.  The walk is bound by the
// latency of its column loads; the atomics of its callers come next (projection bits
// joined before them: 65 us a plane).
#pragma once
#include "k_common.cuh"

namespace libcga {

constexpr uint32_t kWalk = 128;  // positions per step of a warp

// The positions [begin, end) of one warp: u positions in equal contiguous runs
// of whole steps over all warps of the grid.
__device__ __forceinline__ void walk_range(uint32_t u, uint32_t& begin, uint32_t& end) {
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t steps = (u + kWalk - 1) / kWalk;
  const uint32_t per = (steps + warps - 1) / warps;
  const unsigned long long b = (unsigned long long)w * per * kWalk;
  begin = (uint32_t)min(b, (unsigned long long)u);
  end = (uint32_t)min(b + (unsigned long long)per * kWalk, (unsigned long long)u);
}

// f(p, k, x, y, z) for the four positions p + 32 k + lane (k = 0..3) of every
// step [p, p + 128) of [begin, end): arrays of four; `valid` has bit k set when
// the lane's k-th position is below end.  All 32 lanes call f together.
template <typename F>
__device__ __forceinline__ void walk_voxels(const Levels& a, uint32_t begin, uint32_t end, F f) {
  if (begin >= end) return;
  const uint32_t full = 0xffffffffu, lane = threadIdx.x & 31u;
  const uint32_t g = (uint32_t)a.hdr->cnt[1], h = (uint32_t)a.hdr->cnt[2];
  const uint32_t le = 0xffffffffu >> (31u - lane);  // this lane and the ones below
  uint32_t c = warp_search_le(a.ptr1, 0, g - 1, begin);  // column of the last position done
  uint32_t xr = warp_search_le(a.ptr2, 0, h - 1, c);     // its slab
  uint32_t xv = __ldg(a.idx2 + xr), xend = __ldg(a.ptr2 + xr + 1);
  for (uint32_t p = begin; p < end; p += kWalk) {
    uint32_t s[4], x[4], y[4], z[4];
    uint32_t valid = 0;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      const uint32_t e = p + 32 * k + lane, cs = c + 1 + lane + 32 * k;
      s[k] = cs <= g ? __ldg(a.ptr1 + cs) - p : 0xffffffffu;  // at or past p
      z[k] = 0;
      if (e < end) {
        z[k] = __ldg(a.idx0 + e);
        valid |= 1u << k;
      }
    }
    uint32_t cc[4], base = c;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      uint32_t bit = 0;
      // starts ascend: the first 32 k + 32 columns reach past group k
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        if (j <= k && (s[j] >> 5) == k) bit |= 1u << (s[j] & 31u);
      }
      const uint32_t m = __reduce_or_sync(full, bit);
      cc[k] = base + __popc(m & le);
      base += __popc(m);
    }
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      y[k] = ((valid >> k) & 1u) ? __ldg(a.idx1 + cc[k]) : 0u;
      x[k] = xv;
    }
    if (base >= xend && xr + 1 < h) {
      ++xr;
      const uint32_t x0 = xend;
      xv = __ldg(a.idx2 + xr);
      xend = __ldg(a.ptr2 + xr + 1);
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k) x[k] = cc[k] >= x0 ? xv : x[k];
    }
    while (base >= xend) {  // slabs opening inside the step (the sentinel h + 1 is above)
      const uint32_t sl = xr + 1 + lane;
      const uint32_t st = sl <= h ? __ldg(a.ptr2 + sl) : 0xffffffffu;  // first column
      const uint32_t xs = sl < h ? __ldg(a.idx2 + sl) : 0u;
      const uint32_t n = (uint32_t)__popc(__ballot_sync(full, st <= base));
      for (uint32_t i = 0; i < n; ++i) {
        const uint32_t x0 = __shfl_sync(full, st, i);
        xv = __shfl_sync(full, xs, i);
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) x[k] = cc[k] >= x0 ? xv : x[k];
      }
      if (n == 0) break;  // (no slab left: a malformed CGA)
      xr += n;
      xend = n < 32 ? __shfl_sync(full, st, n) : __ldg(a.ptr2 + min(xr + 1, h));
    }
    c = base;
    f(p, valid, x, y, z);
  }
}

// Blocks of 256 threads for a walk over at most `cap` positions: a full wave of
// `per_sm` resident blocks, fewer when the warps would have less than a step.
inline unsigned walk_blocks(uint64_t cap, uint32_t per_sm) {
  const uint64_t steps = (cap + kWalk - 1) / kWalk, b = (steps + 7) / 8;
  const uint64_t most = (uint64_t)device_sm_count() * per_sm;
  return (unsigned)(b < 1 ? 1 : (b < most ? b : most));
}

}  // namespace libcga
