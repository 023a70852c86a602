// The Value (attribute) array of a CGA (Sec. V): one row of uint8 channels
// per stored voxel, in CGA point order.
// Builds by bins sum the rows along with the sort (k_bins.cuh); what follows is the
// way of the other builds (dense grids of many points, and clouds that the general
// sort takes over).
//   k_value_accumulate  each input point finds its voxel by the Sec. V-A
//                       lookup and adds its attributes (or offers its index)
//   k_value_finalize    per voxel: round-half-up mean (sum + k/2) / k of its
//                       k points (Sec. III-B: the colours of the points merged
//                       into one box are averaged), or the first point's row
//   k_merge_values      per voxel of a merge: the row of the input holding
//                       it; in both, the base's (a's) row or the average
//                       (a + b + 1) / 2 (Sec. II-A); any build's inputs
// Sums are integer atomics, 32-bit when no voxel can reach 2^32 (n * 255 <
// 2^32) and 64-bit otherwise, so every result is independent of the order in
// which points arrive.
#include <algorithm>

#include "k_common.cuh"
#include "k_walk.cuh"

namespace libcga {

namespace {

__global__ void k_value_init(uint32_t* scratch, size_t words, uint32_t value,
                             const uint32_t* only_if) {
  if (only_if != nullptr && *only_if == 0) return;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < words; i += stride) {
    scratch[i] = value;
  }
}

template <typename S>
__global__ void k_value_accumulate(Levels a, ValueInput in, void* scratch,
                                   const uint32_t* only_if) {
  if (only_if != nullptr && *only_if == 0) return;
  const uint32_t h = (uint32_t)a.hdr->cnt[2];
  const uint32_t C = in.channels;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < in.n; i += stride) {
    const float* p = in.xyz + 3 * i;
    unsigned long long key;
    if (!point_key<unsigned long long>(__ldg(p), __ldg(p + 1), __ldg(p + 2), in.has_x != 0, in.X,
                                       in.scale, in.off, a.bits, key)) {
      continue;  // the build has recorded the non-finite point
    }
    bool found = false;
    const uint32_t v = rank_of_found(a, h, key, found);
    if (!found) {
      atomicOr(&a.hdr->err, kErrInternal);
      continue;
    }
    if (in.policy == kValueFirst) {
      atomicMin(static_cast<uint32_t*>(scratch) + v, (uint32_t)i);
    } else {
      S* s = static_cast<S*>(scratch) + (size_t)v * (C + 1);
      for (uint32_t c = 0; c < C; ++c) atomicAdd(s + c, (S)__ldg(in.attr + i * C + c));
      atomicAdd(s + C, (S)1);
    }
  }
}

template <typename S>
__global__ void k_value_finalize(Levels a, ValueInput in, const void* scratch, uint8_t* values,
                                 const uint32_t* only_if) {
  if (only_if != nullptr && *only_if == 0) return;
  const uint32_t u = (uint32_t)a.hdr->cnt[0];
  const uint32_t C = in.channels;
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < u; v += stride) {
    if (in.policy == kValueFirst) {
      const uint32_t i = static_cast<const uint32_t*>(scratch)[v];
      for (uint32_t c = 0; c < C; ++c) {
        values[(size_t)v * C + c] = i < in.n ? __ldg(in.attr + (size_t)i * C + c) : (uint8_t)0;
      }
    } else {
      const S* s = static_cast<const S*>(scratch) + (size_t)v * (C + 1);
      const S k = s[C];
      for (uint32_t c = 0; c < C; ++c) {
        values[(size_t)v * C + c] = k > 0 ? (uint8_t)((s[c] + k / 2) / k) : (uint8_t)0;
      }
    }
  }
}

// Where a walk in key order stands in one input of the merge: its slab and column
// ranks at the voxel (x, y).
struct Along {
  uint32_t x, y, slab, col;
};

// The place of voxel (x, y, z) in a, for keys at or past those of `at` (whose ranks
// become the voxel's).  Slab and column ranks grow by at most what x and y do, which
// bounds both searches.
__device__ __forceinline__ uint32_t place_along(const Levels& a, uint32_t h, Along& at, uint32_t x,
                                                uint32_t y, uint32_t z, bool& found) {
  found = false;
  const bool same = x == at.x;
  if (!same) at.slab = lower_bound_u16(a.idx2, at.slab, min(h, at.slab + (x - at.x) + 1), x);
  const uint32_t y0 = at.y;
  at.x = x;
  at.y = y;
  if (at.slab >= h || __ldg(a.idx2 + at.slab) != x) {
    at.col = at.slab < h ? __ldg(a.ptr2 + at.slab) : 0u;
    return 0;
  }
  const uint32_t ye = __ldg(a.ptr2 + at.slab + 1);
  at.col = same ? lower_bound_u16(a.idx1, at.col, min(ye, at.col + (y - y0) + 1), y)
                : lower_bound_u16(a.idx1, __ldg(a.ptr2 + at.slab), ye, y);
  if (at.col >= ye || __ldg(a.idx1 + at.col) != y) return 0;
  const uint32_t zs = __ldg(a.ptr1 + at.col), ze = __ldg(a.ptr1 + at.col + 1);
  const uint32_t p = lower_bound_u16(a.idx0, zs, ze, z);
  found = p < ze && __ldg(a.idx0 + p) == z;
  return p;
}

// The rows of the merged voxels: a walk over m (k_walk.cuh), whose keys ascend, so
// that each voxel's places in both inputs lie a little past the previous step's.  A
// block expanding a tile of m and searching both inputs from their first slab for
// every voxel took 672 us for 20M voxels of 3 channels, this takes 455; 1.8M voxels 107
// and 58, 200k LiDAR voxels at b = 16 86 and 30.  Bound by the latency of the dependent
// loads of two searches a voxel.
constexpr int kMergeValuesPerSm = 5;
__global__ void __launch_bounds__(kThreads, kMergeValuesPerSm)
    k_merge_values(Levels m, Levels a, Levels b, const uint8_t* __restrict__ va,
                   const uint8_t* __restrict__ vb, uint32_t C, int policy,
                   uint8_t* __restrict__ vm) {
  uint32_t begin, end;
  walk_range((uint32_t)m.hdr->cnt[0], begin, end);
  const uint32_t lane = threadIdx.x & 31u, full = 0xffffffffu;
  const uint32_t ha = (uint32_t)a.hdr->cnt[2], hb = (uint32_t)b.hdr->cnt[2];
  Along A{0, 0, 0, 0}, B{0, 0, 0, 0};
  walk_voxels(m, begin, end, [&](uint32_t p, uint32_t valid, const uint32_t* x, const uint32_t* y,
                                 const uint32_t* z) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      Along ta = A, tb = B;
      if ((valid >> k) & 1u) {
        bool fa, fb;
        const uint32_t ia = place_along(a, ha, ta, x[k], y[k], z[k], fa);
        const uint32_t ib = place_along(b, hb, tb, x[k], y[k], z[k], fb);
        uint8_t* out = vm + (size_t)(p + 32 * k + lane) * C;
        for (uint32_t c = 0; c < C; ++c) {
          uint32_t v = 0;
          if (fa && fb) {
            const uint32_t s = __ldg(va + (size_t)ia * C + c), t = __ldg(vb + (size_t)ib * C + c);
            v = policy == kMergeBase ? s : (s + t + 1u) / 2u;
          } else if (fa) {
            v = __ldg(va + (size_t)ia * C + c);
          } else if (fb) {
            v = __ldg(vb + (size_t)ib * C + c);
          }
          out[c] = (uint8_t)v;
        }
      }
      // on from the group's last voxel (of a full group: the walk ends with another)
      A.x = __shfl_sync(full, ta.x, 31);
      A.y = __shfl_sync(full, ta.y, 31);
      A.slab = __shfl_sync(full, ta.slab, 31);
      A.col = __shfl_sync(full, ta.col, 31);
      B.x = A.x;
      B.y = A.y;
      B.slab = __shfl_sync(full, tb.slab, 31);
      B.col = __shfl_sync(full, tb.col, 31);
    }
  });
}

unsigned blocks_for(uint64_t work) {
  return (unsigned)std::min<uint64_t>((std::max<uint64_t>(work, 1) + 255) / 256,
                                      (uint64_t)device_sm_count() * 8);
}

}  // namespace

// 32-bit sums suffice while n points of at most 255 each cannot reach 2^32.
static bool narrow_sums(uint64_t n) { return n * 255ull < (1ull << 32); }

size_t value_scratch_bytes(uint64_t cap, uint32_t channels, int policy) {
  // sized for the wider sums: the count n is not known here
  return (size_t)std::max<uint64_t>(cap, 1) * (policy == kValueFirst ? 4 : 8 * (channels + 1));
}

cudaError_t run_build_values(const Levels& a, const ValueInput& in, void* scratch,
                             uint8_t* values, const uint32_t* only_if, cudaStream_t stream) {
  const bool narrow = in.policy != kValueFirst && narrow_sums(in.n);
  const size_t bytes = narrow ? (size_t)std::max<uint64_t>(a.cap, 1) * 4 * (in.channels + 1)
                              : value_scratch_bytes(a.cap, in.channels, in.policy);
  const uint32_t init = in.policy == kValueFirst ? 0xffffffffu : 0u;
  if (only_if == nullptr) {
    const cudaError_t e = cudaMemsetAsync(scratch, (int)(init & 0xffu), bytes, stream);
    if (e != cudaSuccess) return e;
  } else {
    k_value_init<<<blocks_for(bytes / 16), 256, 0, stream>>>(static_cast<uint32_t*>(scratch),
                                                             bytes / 4, init, only_if);
    count_launch(1);
  }
  if (narrow) {
    k_value_accumulate<uint32_t><<<blocks_for(in.n), 256, 0, stream>>>(a, in, scratch, only_if);
    k_value_finalize<uint32_t><<<blocks_for(a.cap), 256, 0, stream>>>(a, in, scratch, values,
                                                                      only_if);
  } else {
    k_value_accumulate<unsigned long long><<<blocks_for(in.n), 256, 0, stream>>>(a, in, scratch,
                                                                                only_if);
    k_value_finalize<unsigned long long><<<blocks_for(a.cap), 256, 0, stream>>>(a, in, scratch,
                                                                             values, only_if);
  }
  count_launch(2);
  return cudaGetLastError();
}

cudaError_t run_merge_values(const Levels& m, const Levels& a, const Levels& b, const uint8_t* va,
                             const uint8_t* vb, uint32_t channels, int policy, uint8_t* vm,
                             cudaStream_t stream) {
  if (m.cap == 0) return cudaSuccess;
  k_merge_values<<<walk_blocks(m.cap, kMergeValuesPerSm), kThreads, 0, stream>>>(
      m, a, b, va, vb, channels, policy, vm);
  count_launch(1);
  return cudaGetLastError();
}

}  // namespace libcga
