// Perspective projection of a CGA onto an image (Eq. 5-6): every stored voxel
// is moved to the eye's frame, rotated about the y axis (Eq. 6) and divided by
// its depth onto the plane at distance D (Eq. 5); each pixel keeps the voxel
// of least depth, ties to the smaller CGA index.
//   k_perspective         a warp per run of voxels (k_walk.cuh), one 64-bit
//                         atomic minimum per voxel on (depth bits << 32 |
//                         index): a positive float's bits order like the
//                         float, so the minimum is the nearest voxel and then
//                         the smallest index
//   k_perspective_finish  the packed z-buffer to index and depth images
// The arithmetic is one IEEE operation per step in a fixed order (no
// contraction), so the image is the same on every run and device.
#include <algorithm>

#include "k_walk.cuh"

namespace libcga {

namespace {

constexpr int kPerspPerSm = 5;
__global__ void __launch_bounds__(kThreads, kPerspPerSm) k_perspective(Levels a, Camera cam,
                                                                       unsigned long long* zbuf) {
  uint32_t begin, end;
  walk_range((uint32_t)a.hdr->cnt[0], begin, end);
  const uint32_t lane = threadIdx.x & 31u;
  const float half_w = (float)cam.W * 0.5f, half_h = (float)cam.H * 0.5f;
  const float neg_sin = -cam.sin_t;
  walk_voxels(a, begin, end, [&](uint32_t p, uint32_t valid, const uint32_t* x, const uint32_t* y,
                                 const uint32_t* z) {
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
      if (!((valid >> k) & 1u)) continue;
      const float sx = __fsub_rn((float)x[k], cam.eye[0]);
      const float sy = __fsub_rn((float)y[k], cam.eye[1]);
      const float sz = __fsub_rn((float)z[k], cam.eye[2]);
      const float xr = __fmaf_rn(cam.cos_t, sx, __fmul_rn(neg_sin, sz));
      const float zr = __fmaf_rn(cam.sin_t, sx, __fmul_rn(cam.cos_t, sz));
      if (!(zr > 0.0f)) continue;  // at or behind the eye
      const float px = __fdiv_rn(__fmul_rn(cam.D, xr), zr);
      const float py = __fdiv_rn(__fmul_rn(cam.D, sy), zr);
      const float fu = floorf(__fadd_rn(px, half_w)), fv = floorf(__fadd_rn(py, half_h));
      if (!(fu >= 0.0f && fu < (float)cam.W && fv >= 0.0f && fv < (float)cam.H)) continue;
      const size_t pix = (size_t)fv * cam.W + (size_t)fu;
      atomicMin(zbuf + pix, ((unsigned long long)__float_as_uint(zr) << 32) |
                                (unsigned long long)(p + 32 * k + lane));
    }
  });
}

__global__ void k_perspective_finish(const unsigned long long* __restrict__ zbuf, uint64_t npix,
                                     uint32_t* __restrict__ index, float* __restrict__ depth) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < npix; i += stride) {
    const unsigned long long v = zbuf[i];
    index[i] = (uint32_t)v;
    depth[i] = v == ~0ull ? __int_as_float(0x7f800000) : __uint_as_float((uint32_t)(v >> 32));
  }
}

}  // namespace

cudaError_t run_perspective(const Levels& a, const Camera& cam, unsigned long long* zbuf,
                            uint32_t* index, float* depth, cudaStream_t stream) {
  const uint64_t npix = (uint64_t)cam.W * cam.H;
  cudaError_t e = cudaMemsetAsync(zbuf, 0xff, npix * sizeof(unsigned long long), stream);
  if (e != cudaSuccess) return e;
  if (a.cap > 0) {
    k_perspective<<<walk_blocks(a.cap, kPerspPerSm), kThreads, 0, stream>>>(a, cam, zbuf);
  }
  const unsigned blocks = (unsigned)std::min<uint64_t>((npix + 255) / 256,
                                                       (uint64_t)device_sm_count() * 8);
  k_perspective_finish<<<blocks, 256, 0, stream>>>(zbuf, npix, index, depth);
  count_launch(a.cap > 0 ? 2 : 1);
  return cudaGetLastError();
}

}  // namespace libcga
