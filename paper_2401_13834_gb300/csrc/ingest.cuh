// Reading blocks: 16 samples of a channel-major row, and the 64 x 64 tiles of
// time-major blocks. Included by the kernels that bring blocks into a beam's
// buffer (kernels.cuh, floatpath.cu).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace {

// 16 samples t .. t + 15 of `row`, those outside [0, n) zero. The row lies in a
// buffer [base, end); aligned words inside it are read whole and shifted
// into place, so that a row may start at any byte.
__device__ __forceinline__ uint4 ft_chunk(const uint8_t* __restrict__ base, const uint8_t* __restrict__ end,
                                          const uint8_t* __restrict__ row, int64_t t, int64_t n) {
  const uint8_t* p = row + t;
  if (t >= 0 && t + 16 <= n) {
    const int a = (int)((uintptr_t)p & 15);
    if (a == 0) return __ldg(reinterpret_cast<const uint4*>(p));
    const uint8_t* q = p - (a & 3);
    if (q >= base && q + 20 <= end) {
      const uint32_t* w = reinterpret_cast<const uint32_t*>(q);
      const uint32_t w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2), w3 = __ldg(w + 3), w4 = __ldg(w + 4);
      const int s = 8 * (a & 3);
      return make_uint4(__funnelshift_r(w0, w1, s), __funnelshift_r(w1, w2, s), __funnelshift_r(w2, w3, s),
                        __funnelshift_r(w3, w4, s));
    }
  }
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (t + i >= 0 && t + i < n) w[i >> 2] |= (uint32_t)p[i] << (8 * (i & 3));
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Stores samples t .. t + 15 (those in [0, n)) at the 16-byte aligned d.
__device__ __forceinline__ void store16(uint8_t* d, uint4 v, int64_t t, int64_t n) {
  if (t >= 0 && t + 16 <= n) {
    *reinterpret_cast<uint4*>(d) = v;
    return;
  }
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 16; ++i)
    if (t + i >= 0 && t + i < n) d[i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
}

// How time-major rows of nchan bytes from `src` on can be read: 16 bytes at a
// time (2), 4 (1) or 1 (0).
inline int tf_load_form(const void* src, int nchan) {
  const int a = (int)((uintptr_t)src & 15);
  return nchan % 16 == 0 && a == 0 ? 2 : nchan % 4 == 0 && (a & 3) == 0 ? 1 : 0;
}

// This thread's 16 bytes of the 64-time x 64-channel byte tile (times t0..,
// channels c0..) of a time-major block [t][nchan]: time t0 + tid / 4,
// channels c0 + 16 (tid % 4) ..; zero outside the block. 256 threads.
__device__ __forceinline__ uint4 tf_tile_chunk(const uint8_t* __restrict__ src, int64_t t0, int64_t n, int c0,
                                               int nchan, int ld) {
  const int r = threadIdx.x >> 2, q = threadIdx.x & 3;
  const int64_t t = t0 + r;
  const int c = c0 + 16 * q;
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (t >= 0 && t < n) {
    const uint8_t* sp = src + t * nchan + c;
    if (ld == 2 && c + 16 <= nchan) {
      v = __ldg(reinterpret_cast<const uint4*>(sp));
    } else if (ld) {   // channels in fours
      const uint32_t* wp = reinterpret_cast<const uint32_t*>(sp);
      if (c < nchan) v.x = __ldg(wp);
      if (c + 4 < nchan) v.y = __ldg(wp + 1);
      if (c + 8 < nchan) v.z = __ldg(wp + 2);
      if (c + 12 < nchan) v.w = __ldg(wp + 3);
    } else {
      uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (c + i < nchan) w[i >> 2] |= (uint32_t)sp[i] << (8 * (i & 3));
      v = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  return v;
}

// Column cc of a tile, times 16 pq .. 16 pq + 15, as four little-endian words.
__device__ __forceinline__ void tf_column(const uint8_t (*tile)[80], int cc, int pq, uint32_t w[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    w[i] = (uint32_t)tile[16 * pq + 4 * i][cc] | ((uint32_t)tile[16 * pq + 4 * i + 1][cc] << 8) |
           ((uint32_t)tile[16 * pq + 4 * i + 2][cc] << 16) | ((uint32_t)tile[16 * pq + 4 * i + 3][cc] << 24);
}

}  // namespace
