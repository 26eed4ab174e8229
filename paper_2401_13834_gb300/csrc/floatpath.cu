// The float path (sm_103a): per-channel normalisation (Sec. 2.1) before the
// sub-band de-dispersion (Sec. 2.3) and the boxcar matched filter (Sec. 2.4,
// Eq. 5), for plans with a tx_norm mode.
//
// Per block of a beam:
//   k_chan_sums_*   exact sums of x and x^2 per channel over the block's T new samples
//   k_chan_weights  mu_c, sigma_c (population), weight w_c = 1/sigma_c or 1/sigma_c^2
//   k_norm_ingest_* x' = (float(x) - mu_c) * w_c into the beam's float32 circular buffer
//                   behind the carried tail (which keeps its own block's normalisation)
//   k_stage1_f32    P[k][s][t] = sum_{c in s} x'[c][t + d1[k][c]]  (FP32, channels in order)
//   k_stage2_pipe32 D[d][t]    = sum_s P[k(d)][s][t + d2[d][s]]     (FP32, sub-bands in order),
//                   with per-tile sums of D and D^2 (stage2_pipe32.cuh)
//   k_stats_f32     mu_d, sigma_d of D over [0, T) in double (block or running)
//   k_boxcar_f32    compensated (TwoSum) prefix sums of D per tile as float (hi, lo) pairs,
//                   window sums B_W = C[t + W] - C[t], S/N = (B_W - W mu_d) / (sigma_d sqrt W)
// The float path trades the integer path's packed sums for arithmetic on
// normalised data.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "device.cuh"
#include "ingest.cuh"
#include "stage2_pipe32.cuh"
#include "tx_internal.h"

using namespace tx;

#define TX_CUDA(expr)                                                               \
  do {                                                                              \
    cudaError_t e_ = (expr);                                                        \
    if (e_ != cudaSuccess) {                                                        \
      set_error("%s failed: %s", #expr, cudaGetErrorString(e_));                    \
      return TX_ERR_CUDA;                                                           \
    }                                                                               \
  } while (0)

namespace {

constexpr int kThreads = 256;
constexpr int kSumBytes = 16384;  // bytes of a channel-major row per block of the channel sums

// ---- channel statistics -----------------------------------------------------
// S[c] = (sum x, sum x^2) over samples t < n of channel c; block in the plan's
// layout (FT rows of `pitch` bytes, or TF rows of nchan bytes). Atomic integer
// adds: exact and order-free. Both read four samples of a channel per
// instruction (dp4a): with one byte per load and one per store of the samples, a
// MeerKAT-L block took 0.83 ms to normalise (now 0.31), and 320 channels x 14336
// samples 0.29 ms on the eight SMs that summed them (now 0.02).
//
// Channel-major: one block per (row, kSumBytes bytes of it).
__global__ void __launch_bounds__(kThreads) k_chan_sums_ft(const uint8_t* __restrict__ blk, int64_t n, int64_t pitch,
                                                            unsigned long long* __restrict__ S) {
  pdl_wait();
  pdl_trigger();
  const int c = blockIdx.y;
  const uint8_t* row = blk + (int64_t)c * pitch;
  const uint8_t* end = blk + (int64_t)gridDim.y * pitch;
  const int64_t t0 = (int64_t)blockIdx.x * kSumBytes, t1 = min(n, t0 + kSumBytes);
  unsigned s1 = 0, s2 = 0;   // at most 64 samples a thread
#pragma unroll
  for (int i = 0; i < kSumBytes / 16 / kThreads; ++i) {
    const int64_t t = t0 + 16 * (threadIdx.x + i * kThreads);
    if (t >= t1) break;
    const uint4 v = ft_chunk(blk, end, row, t, t1);
    s1 = __dp4a(v.x, 0x01010101u, __dp4a(v.y, 0x01010101u, __dp4a(v.z, 0x01010101u, __dp4a(v.w, 0x01010101u, s1))));
    s2 = __dp4a(v.x, v.x, __dp4a(v.y, v.y, __dp4a(v.z, v.z, __dp4a(v.w, v.w, s2))));
  }
  __shared__ unsigned r1[kThreads / 32], r2[kThreads / 32];
  s1 = __reduce_add_sync(0xffffffffu, s1);
  s2 = __reduce_add_sync(0xffffffffu, s2);
  if ((threadIdx.x & 31) == 0) { r1[threadIdx.x >> 5] = s1; r2[threadIdx.x >> 5] = s2; }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long a = 0, b = 0;
    for (int w = 0; w < kThreads / 32; ++w) { a += r1[w]; b += r2[w]; }
    atomicAdd(S + 2 * c, a);
    atomicAdd(S + 2 * c + 1, b);
  }
}

// Time-major: blocks of 256 channels x `chunk` times (a multiple of 16, at most
// kSumBytes). Thread q + 64 p takes channels 4 q .. 4 q + 3 at times 4 p .. 4 p +
// 3 of every 16; four rows' words are transposed to a word per channel.
__global__ void __launch_bounds__(kThreads) k_chan_sums_tf(const uint8_t* __restrict__ blk, int nchan, int64_t n,
                                                            int chunk, int words, unsigned long long* __restrict__ S) {
  __shared__ unsigned r1[4][kThreads], r2[4][kThreads];
  pdl_wait();
  pdl_trigger();
  const int q = threadIdx.x & 63, p = threadIdx.x >> 6;
  const int c = blockIdx.y * 256 + 4 * q;
  const int64_t t0 = (int64_t)blockIdx.x * chunk, t1 = min(n, t0 + chunk);
  unsigned s1[4] = {0u, 0u, 0u, 0u}, s2[4] = {0u, 0u, 0u, 0u};
#pragma unroll 2
  for (int64_t t = t0 + 4 * p; t < t1; t += 16) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      w[i] = 0u;
      if (t + i < t1) {
        const uint8_t* s = blk + (t + i) * nchan + c;
        if (words) {
          if (c < nchan) w[i] = __ldg(reinterpret_cast<const uint32_t*>(s));
        } else {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (c + k < nchan) w[i] |= (uint32_t)s[k] << (8 * k);
        }
      }
    }
    const uint32_t a0 = __byte_perm(w[0], w[1], 0x5140), a1 = __byte_perm(w[0], w[1], 0x7362);
    const uint32_t b0 = __byte_perm(w[2], w[3], 0x5140), b1 = __byte_perm(w[2], w[3], 0x7362);
    const uint32_t x[4] = {__byte_perm(a0, b0, 0x5410), __byte_perm(a0, b0, 0x7632), __byte_perm(a1, b1, 0x5410),
                           __byte_perm(a1, b1, 0x7632)};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s1[k] = __dp4a(x[k], 0x01010101u, s1[k]);
      s2[k] = __dp4a(x[k], x[k], s2[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    r1[p][4 * q + k] = s1[k];
    r2[p][4 * q + k] = s2[k];
  }
  __syncthreads();
  const int ch = blockIdx.y * 256 + threadIdx.x;
  if (ch >= nchan) return;
  unsigned long long a = 0, b = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) { a += r1[i][threadIdx.x]; b += r2[i][threadIdx.x]; }
  atomicAdd(S + 2 * ch, a);
  atomicAdd(S + 2 * ch + 1, b);
}

// (mu_c, w_c) as floats from the exact sums over n samples: mu = S1 / n,
// var = (n S2 - S1^2) / n^2 with an exact 128-bit numerator, sigma = sqrt(var),
// w = 1 / sigma (unit variance) or 1 / var (weights by the reciprocal of the
// variance), 0 when sigma = 0.
__global__ void k_chan_weights(const unsigned long long* __restrict__ S, int nchan, int64_t n, int norm,
                               float2* __restrict__ muw) {
  pdl_wait();
  pdl_trigger();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nchan) return;
  const unsigned long long s1 = S[2 * c], s2 = S[2 * c + 1];
  const double mu = __ddiv_rn((double)s1, (double)n);
  const unsigned __int128 num = (unsigned __int128)(unsigned long long)n * s2 - (unsigned __int128)s1 * s1;
  const double hi = (double)(unsigned long long)(num >> 64), lo = (double)(unsigned long long)num;
  const double var = __ddiv_rn(__dadd_rn(__dmul_rn(hi, 18446744073709551616.0), lo), __dmul_rn((double)n, (double)n));
  double w = 0.0;
  if (var > 0.0) w = norm == TX_NORM_UNIT ? __ddiv_rn(1.0, sqrt(var)) : __ddiv_rn(1.0, var);
  muw[c] = make_float2(__double2float_rn(mu), __double2float_rn(w));
}

__device__ __forceinline__ float norm_sample(unsigned x, float2 mw) {
  return __fmul_rn(__fsub_rn((float)x, mw.x), mw.y);
}

// x' of samples t < n into ring[c][(pos0 + t) mod R], four samples of the ring's
// 16-byte grid per store (R is a multiple of 64, so none straddles the wrap).
// d: the position of sample t, a multiple of 4.
__device__ __forceinline__ void norm_store4(float* __restrict__ row, int64_t R, int64_t pos, uint32_t x, int64_t t,
                                            int64_t n, float2 mw) {
  if (pos >= R) pos -= R;
  const float v[4] = {norm_sample(x & 255u, mw), norm_sample((x >> 8) & 255u, mw), norm_sample((x >> 16) & 255u, mw),
                      norm_sample(x >> 24, mw)};
  if (t >= 0 && t + 4 <= n) {
    *reinterpret_cast<float4*>(row + pos) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (t + i >= 0 && t + i < n) row[pos + i] = v[i];
  }
}

// Channel-major rows, one per blockIdx.y.
__global__ void __launch_bounds__(kThreads) k_norm_ingest_ft(const uint8_t* __restrict__ src, int64_t n, int64_t pitch,
                                                              float* __restrict__ ring, int64_t R, int64_t pos0,
                                                              const float2* __restrict__ muw) {
  pdl_wait();
  pdl_trigger();
  const int c = blockIdx.y, shift = (int)(pos0 & 3);
  const float2 mw = muw[c];
  const uint8_t* row = src + (int64_t)c * pitch;
  float* out = ring + (int64_t)c * R;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; 4 * i - shift < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = 4 * i - shift;
    uint32_t x = 0u;
    if (t >= 0 && t + 4 <= n && ((uintptr_t)(row + t) & 3) == 0) {
      x = __ldg(reinterpret_cast<const uint32_t*>(row + t));
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (t + k >= 0 && t + k < n) x |= (uint32_t)__ldg(row + t + k) << (8 * k);
    }
    norm_store4(out, R, pos0 + t, x, t, n, mw);
  }
}

// Time-major blocks, kNormTiles 64-time x 64-channel byte tiles per block (all
// loads in flight first) through shared memory, 16 lanes to a channel's 64
// times. ld: see tf_load_form.
constexpr int kNormTiles = 2;
__global__ void __launch_bounds__(kThreads) k_norm_ingest_tf(const uint8_t* __restrict__ src, int nchan, int64_t n,
                                                              float* __restrict__ ring, int64_t R, int64_t pos0, int ld,
                                                              const float2* __restrict__ muw) {
  __shared__ uint32_t tile[kNormTiles][64][17];   // a time's 64 channels, padded by a word
  pdl_wait();
  pdl_trigger();
  const int c0 = blockIdx.y * 64;
  const int64_t t0 = (int64_t)blockIdx.x * kNormTiles * 64 - (pos0 & 3);
  uint4 v[kNormTiles];
#pragma unroll
  for (int i = 0; i < kNormTiles; ++i) v[i] = tf_tile_chunk(src, t0 + 64 * i, n, c0, nchan, ld);
#pragma unroll
  for (int i = 0; i < kNormTiles; ++i) {
    uint32_t* w = &tile[i][threadIdx.x >> 2][4 * (threadIdx.x & 3)];
    w[0] = v[i].x;
    w[1] = v[i].y;
    w[2] = v[i].z;
    w[3] = v[i].w;
  }
  __syncthreads();
  const int l = threadIdx.x & 15;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int cc = (threadIdx.x >> 4) + 16 * k, c = c0 + cc;
    if (c >= nchan) break;
    const float2 mw = muw[c];
    float* row = ring + (int64_t)c * R;
#pragma unroll
    for (int i = 0; i < kNormTiles; ++i) {
      const int64_t t = t0 + 64 * i + 4 * l;
      if (t >= n) break;
      uint32_t x = 0u;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        x |= (uint32_t)reinterpret_cast<const uint8_t*>(tile[i][4 * l + j])[cc] << (8 * j);
      norm_store4(row, R, pos0 + t, x, t, n, mw);
    }
  }
}

// ---- de-dispersion ----------------------------------------------------------------
// Stage 1: P[k][s][t] = sum_{c in s} x'[c][t + d1[k][c]], channels one after the
// other (the sum order, and so every bit of the result, is part of the path).
// Bound: shared memory, 4 bytes per sample-add that needs its own load (7.1 ms
// for the 69e9 sample-adds of a MeerKAT-L block at 39.1 TB/s). A warp sums
// four consecutive coarse DMs, and where neighbours have the same delay in a
// channel they add the same registers: a quarter of the loads of a MeerKAT-L
// block go that way.
//
// Persistent blocks walk the items (unit u = blockIdx.x + i gridDim.x) in
// chunks of up to 16 channels through kF1Stages stages, without block-wide
// barriers: the last warp bulk-copies (TMA) a chunk's windows of the ring, one
// per lane (two where a window wraps the ring's end), and its offset table
// (mbarriers full / empty); the others keep their four coarse DMs' sums in
// registers over an item's chunks, VW outputs per lane. Tiles of 512 outputs
// make a warp's part 256 outputs, 8 independent loads in flight per coarse DM,
// for up to 40 coarse DMs on 20 warps.
// One block per item that staged all its channels, then summed, took 12.57
// ms on that block; this takes 7.59 ms with shared memory and issue both 80%
// busy (every load taken: 8.30; 30 warps, which spill: 12.5; predicated loads
// instead of branches, which keep their shared-memory slots: 8.25). Waits are
// bounded as in k_stage2_pipe.
struct F1Args {
  const float* ring;
  const Stage1Item* items;
  const int32_t* chunks;
  const uint32_t* tab;
  const int32_t* abase;    // [nk][nsub]
  float* P;
  double* run;             // the beam's running statistics, then its count of given-up waits
  int64_t R, start, Pp;
  int32_t m, nsub, ndm, nitems;
  int32_t phase;           // which of a chunk's tables
  uint32_t polls;
};

struct F1Shared {
  uint64_t full[kF1Stages], empty[kF1Stages];
  int abort_flag;
};

// One item's sums by one consumer warp; false when a wait gave up.
template <int VW>
__device__ __forceinline__ bool f1_consume(const F1Args& a, F1Shared& sh, const float* stages, const Stage1Item& it,
                                           int warp, int lane, int& st, uint32_t& par) {
  constexpr int PARTS = kF1Tile / 32 / VW;
  const int quads = (it.ke - it.kb + kF1Quad - 1) / kF1Quad;
  const bool busy = warp < quads * PARTS;
  const int quad = warp / PARTS, j0 = (warp - quad * PARTS) * 32 * VW + lane;   // this lane's first output
  const int k0 = it.kb + quad * kF1Quad;
  float acc[kF1Quad][VW];
#pragma unroll
  for (int i = 0; i < kF1Quad; ++i)
#pragma unroll
    for (int v = 0; v < VW; ++v) acc[i][v] = 0.f;
  for (int left = a.m; left > 0; left -= kF1Chan) {
    const int nc = min(left, kF1Chan);
    if (!mbar_wait_warp(&sh.full[st], par, a.polls, &sh.abort_flag)) return false;
    if (busy) {
      const float* r = stages + (size_t)st * kF1StageWords + j0;
      const uint2* t = reinterpret_cast<const uint2*>(stages + (size_t)st * kF1StageWords + kF1Chan * kF1RawWords) +
                       quad * kF1Chan;
      auto channel = [&](uint2 o) {
        float x[VW];
        uint32_t at = 0u;
#pragma unroll
        for (int i = 0; i < kF1Quad; ++i) {
          const uint32_t w = i < 2 ? o.x : o.y;
          const uint32_t oi = (i & 1) ? w >> 16 : w & 0xFFFFu;
          if (i == 0 || oi != at) {   // a delay of its own
#pragma unroll
            for (int v = 0; v < VW; ++v) x[v] = r[oi + 32 * v];
          }
          at = oi;
#pragma unroll
          for (int v = 0; v < VW; ++v) acc[i][v] = __fadd_rn(acc[i][v], x[v]);
        }
      };
      int c = 0;
      for (; c + 1 < nc; c += 2) {
        const uint4 o = *reinterpret_cast<const uint4*>(t + c);
        channel(make_uint2(o.x, o.y));
        channel(make_uint2(o.z, o.w));
      }
      if (c < nc) channel(t[c]);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.empty[st]);
    if (++st == kF1Stages) { st = 0; par ^= 1u; }
  }
#pragma unroll
  for (int i = 0; i < kF1Quad; ++i) {
    if (!busy || k0 + i >= it.ke) continue;
    const size_t row = (size_t)(k0 + i) * a.nsub + it.s;
    const int64_t j = (int64_t)it.tau0 - __ldg(a.abase + row) + j0;
    float* prow = a.P + row * a.Pp;
#pragma unroll
    for (int v = 0; v < VW; ++v)
      if (j + 32 * v >= 0 && j + 32 * v < a.Pp) prow[j + 32 * v] = acc[i][v];
  }
  return true;
}

constexpr int kF1Threads = (kF1Consumers + 1) * 32;

__global__ void __launch_bounds__(kF1Threads, 1) k_stage1_f32(const F1Args a) {
  extern __shared__ __align__(16) float smf[];
  __shared__ __align__(8) F1Shared sh;
  pdl_wait();
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int)blockIdx.x >= a.nitems) return;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kF1Stages; ++i) {
      mbar_init(&sh.full[i], 1);
      mbar_init(&sh.empty[i], kF1Consumers);
    }
    sh.abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();   // barriers initialised: the only block-wide barrier
  volatile int* abort = &sh.abort_flag;
  auto give_up = [&]() {
    if (atomicExch(&sh.abort_flag, 1) == 0) record_give_up(a);
  };
  int st = 0;
  uint32_t par = 0u;

  if (warp == kF1Consumers) {
    // --------------------------------------------------------- the issuing warp
    // (a chunk's record, and an item's descriptor, are loaded one ahead: the
    // copies never wait for a dependent global load)
    int64_t q = 0;
    Stage1Item it = a.items[blockIdx.x], nx = it;
    int u = blockIdx.x, ch = 0;
    int rec = __ldg(a.chunks + (size_t)it.tab * kF1Rec + lane);
    while (true) {
      if (ch == 0 && u + (int)gridDim.x < a.nitems) nx = a.items[u + gridDim.x];
      const bool more = ch + 1 < it.pad1 || u + (int)gridDim.x < a.nitems;
      const int nrec = ch + 1 < it.pad1 ? it.tab + ch + 1 : nx.tab;
      int rn = 0;
      if (more) rn = __ldg(a.chunks + (size_t)nrec * kF1Rec + lane);
      const int words = (3 + kF1Tile + it.span + 3) & ~3;   // a window: misalignment, tile, spread
      const int cn = __shfl_sync(0xffffffffu, rec, 0), tw = __shfl_sync(0xffffffffu, rec, 1);
      const int to = __shfl_sync(0xffffffffu, rec, 2), dl = __shfl_sync(0xffffffffu, rec, 8 + (lane & 15));
      const int c0 = cn >> 5, nc = cn & 31;
      if (q >= kF1Stages && !mbar_wait_warp(&sh.empty[st], par ^ 1u, a.polls, abort)) {
        give_up();
        break;
      }
      float* dst = smf + (size_t)st * kF1StageWords;
      if (lane == 0) mbar_expect_tx(&sh.full[st], (uint32_t)(nc * words + tw) * 4u);
      __syncwarp();
      fence_proxy_async();
      if (lane < nc) {
        int64_t p = a.start + it.tau0 + dl;
        while (p >= a.R) p -= a.R;
        const int64_t pa = p & ~(int64_t)3;
        const float* row = a.ring + (size_t)(c0 + lane) * a.R;
        float* d = dst + lane * kF1RawWords;
        // in pieces where the window wraps the ring's end (a short ring more than once)
        int64_t from = pa;
        for (int done = 0; done < words;) {
          const int len = (int)min((int64_t)(words - done), a.R - from);
          bulk_g2s(d + done, row + from, (uint32_t)len * 4u, &sh.full[st]);
          done += len;
          from = 0;
        }
      }
      if (lane == 31)
        bulk_g2s(dst + kF1Chan * kF1RawWords, a.tab + (size_t)to * 4 + (size_t)a.phase * tw, (uint32_t)tw * 4u,
                 &sh.full[st]);
      ++q;
      if (++st == kF1Stages) { st = 0; par ^= 1u; }
      if (!more) break;
      rec = rn;
      if (++ch == it.pad1) {
        ch = 0;
        u += gridDim.x;
        it = nx;
      }
    }
    if (lane == 0) {
      // copies still in flight complete before the block's shared memory is released
      for (int64_t r = q > kF1Stages ? q - kF1Stages : 0; r < q; ++r)
        mbar_wait(&sh.full[(int)(r % kF1Stages)], (uint32_t)((r / kF1Stages) & 1), kMbarPolls);
    }
    return;
  }

  // ------------------------------------------------------------------ consumers
  for (int u = blockIdx.x; u < a.nitems; u += gridDim.x) {
    const Stage1Item it = a.items[u];
    bool ok = false;
    switch (it.pad2) {
      case 8: ok = f1_consume<8>(a, sh, smf, it, warp, lane, st, par); break;
      case 4: ok = f1_consume<4>(a, sh, smf, it, warp, lane, st, par); break;
      default: ok = f1_consume<2>(a, sh, smf, it, warp, lane, st, par); break;
    }
    if (!ok) {
      give_up();
      return;
    }
  }
}

// mu_d = sum D / T, var_d = sum D^2 / T - mu_d^2 (at least 0), or their running
// update; (mu_d, sigma_d) to ms[d].
__global__ void k_stats_f32(const double2* __restrict__ part, int ntile, int ndm, int64_t T, int running, double lam,
                            double* __restrict__ run, double2* __restrict__ ms) {
  const int d = blockIdx.x * blockDim.x + threadIdx.x;
  if (d >= ndm) return;
  double s1 = 0.0, s2 = 0.0;
  for (int i = 0; i < ntile; ++i) {
    const double2 v = part[(size_t)d * ntile + i];
    s1 += v.x;
    s2 += v.y;
  }
  double mu = s1 / (double)T;
  double var = fmax(s2 / (double)T - mu * mu, 0.0);
  if (running) {
    double* r = run + (size_t)d * 2;
    if (r[1] < 0.0) {
      r[0] = mu;
      r[1] = var;
    } else {
      mu = (1.0 - lam) * r[0] + lam * mu;
      var = (1.0 - lam) * r[1] + lam * var;
      r[0] = mu;
      r[1] = var;
    }
  }
  ms[d] = make_double2(mu, sqrt(var));
}

// ---- boxcar (Eq. 5) -------------------------------------------------------------
// Error-free sum of two floats (Knuth's TwoSum): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
// (s, c) += x, compensated: s + c carries the running sum to about twice the
// float precision (TwoSum of s and x, the rounding error added into c).
__device__ __forceinline__ void comp_add(float& s, float& c, float x) {
  float e;
  two_sum(s, x, s, e);
  c = __fadd_rn(c, e);
}

// One block per unit (fine DM d, tile of kBoxTile outputs). The window
// D[t0 + i], i < N = n + W_max - 1, is turned into compensated prefix sums
// C[i] = (hi_i, lo_i), hi_i + lo_i = D[t0] + ... + D[t0 + i - 1] to about twice
// float precision (TwoSum at every add, also across threads and warps), so that
//   B_W[t] = (hi[t+W] - hi[t]) + (lo[t+W] - lo[t])
// takes FP32 operations only and each difference of two floats is rounded
// once, relative to itself. Eq. 5 then subtracts W mu_d as a float pair (from
// double) and scales by 1 / (sigma_d sqrt W): S/N = ((dhi - Wmu_hi) + (dlo -
// Wmu_lo)) * inv (0 when sigma_d = 0). Outputs as the integer path's.
__global__ void __launch_bounds__(kThreads) k_boxcar_f32(const float* __restrict__ D, int64_t Dp, int64_t T,
                                                          int tileL, int ntile3, const double2* __restrict__ ms,
                                                          const int32_t* __restrict__ widths, int nw, int wmax,
                                                          int mode, float gamma, float* __restrict__ outf,
                                                          uint8_t* __restrict__ outw, tx_cand* __restrict__ cands,
                                                          unsigned long long* __restrict__ ncand, int64_t max_cands) {
  extern __shared__ float2 H[];   // [tileL + wmax]: the window, then its prefix sums (hi, lo)
  __shared__ float2 wtot[kThreads / 32];
  __shared__ int32_t sW[kMaxWidths];
  __shared__ float sInv[kMaxWidths], sMh[kMaxWidths], sMl[kMaxWidths];
  const int unit = blockIdx.x;
  const int d = unit / ntile3, tile = unit - d * ntile3;
  const int64_t t0 = (int64_t)tile * tileL;
  const int n = (int)min((int64_t)tileL, T - t0);
  const int N = n + wmax - 1;
  const double2 m = ms[d];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < nw) {
    const int W = widths[threadIdx.x];
    const double wmu = (double)W * m.x;
    const float h = __double2float_rn(wmu);
    sW[threadIdx.x] = W;
    sMh[threadIdx.x] = h;
    sMl[threadIdx.x] = __double2float_rn(wmu - (double)h);
    sInv[threadIdx.x] = m.y > 0.0 ? __double2float_rn(1.0 / (m.y * sqrt((double)W))) : 0.f;
  }
  const float* row = D + (size_t)d * Dp + t0;
  for (int i = threadIdx.x; i < N; i += kThreads) H[i].x = row[i];
  __syncthreads();
  // exclusive compensated scan of H[0..N] in place (element N enters no used sum)
  const int E = (N + 1 + kThreads - 1) / kThreads;
  const int beg = threadIdx.x * E, end = min(beg + E, N + 1);
  float ls = 0.f, lc = 0.f;                                 // this thread's elements
  for (int i = beg; i < end && i < N; ++i) comp_add(ls, lc, H[i].x);
  float xs = ls, xc = lc;                                   // inclusive scan over the warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float ys = __shfl_up_sync(0xffffffffu, xs, o), yc = __shfl_up_sync(0xffffffffu, xc, o);
    if (lane >= o) {
      float e;
      two_sum(ys, xs, xs, e);
      xc = __fadd_rn(__fadd_rn(xc, yc), e);
    }
  }
  if (lane == 31) wtot[warp] = make_float2(xs, xc);
  // this thread's exclusive prefix within the warp: the inclusive one less its own part
  const float ps = __shfl_up_sync(0xffffffffu, xs, 1), pc = __shfl_up_sync(0xffffffffu, xc, 1);
  __syncthreads();
  float s = 0.f, c = 0.f;
  for (int w = 0; w < warp; ++w) {
    comp_add(s, c, wtot[w].x);
    c = __fadd_rn(c, wtot[w].y);
  }
  if (lane > 0) {
    comp_add(s, c, ps);
    c = __fadd_rn(c, pc);
  }
  for (int i = beg; i < end; ++i) {
    const float v = i < N ? H[i].x : 0.f;
    H[i] = make_float2(s, c);
    comp_add(s, c, v);
  }
  __syncthreads();
  // outputs tid + 256 r, RR at once: a width's constants are read from shared
  // memory once for them (the MeerKAT-L plane: 1.87 -> 1.52 ms)
  constexpr int RR = 8;
  for (int i0 = threadIdx.x; i0 - (int)threadIdx.x < n; i0 += RR * kThreads) {
    float2 c0[RR];
    float best[RR];
    int bw[RR];
#pragma unroll
    for (int r = 0; r < RR; ++r) {
      const int i = i0 + r * kThreads;
      c0[r] = i < n ? H[i] : make_float2(0.f, 0.f);
      best[r] = -INFINITY;
      bw[r] = 0;
    }
#pragma unroll 1
    for (int w = 0; w < nw; ++w) {
      const float2* Hw = H + i0 + sW[w];
      const float mh = sMh[w], ml = sMl[w], inv = sInv[w];
      float* o = outf + ((size_t)d * nw + w) * T + t0 + i0;   // cube
#pragma unroll
      for (int r = 0; r < RR; ++r) {
        if (i0 + r * kThreads >= n) break;
        const float2 c1 = Hw[r * kThreads];
        const float B = __fadd_rn(__fsub_rn(__fsub_rn(c1.x, c0[r].x), mh), __fsub_rn(__fsub_rn(c1.y, c0[r].y), ml));
        const float snr = __fmul_rn(B, inv);
        if (mode == TX_OUT_CUBE) o[r * kThreads] = snr;
        else if (snr > best[r]) { best[r] = snr; bw[r] = w; }
      }
    }
#pragma unroll
    for (int r = 0; r < RR; ++r) {
      const int i = i0 + r * kThreads;
      if (mode == TX_OUT_PLANE) {
        if (i < n) {
          outf[(size_t)d * T + t0 + i] = best[r];
          outw[(size_t)d * T + t0 + i] = (uint8_t)bw[r];
        }
      } else if (mode == TX_OUT_CANDS) {
        const bool hit = i < n && best[r] >= gamma;
        const unsigned hits = __ballot_sync(0xffffffffu, hit);
        if (!hits) continue;
        const int leader = __ffs(hits) - 1;
        unsigned long long base = 0;
        if (lane == leader) base = atomicAdd(ncand, (unsigned long long)__popc(hits));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (hit) {
          const unsigned long long idx = base + __popc(hits & ((1u << lane) - 1u));
          if (idx < (unsigned long long)max_cands) {
            tx_cand rec;
            rec.dm_index = d;
            rec.t = (int32_t)(t0 + i);
            rec.w_index = bw[r];
            rec.snr = best[r];
            cands[idx] = rec;
          }
        }
      }
    }
  }
}

inline int64_t mod(int64_t a, int64_t r) { return ((a % r) + r) % r; }

// Channel sums, weights and the normalised samples of n samples at ring
// position pos (src in the plan's layout, FT rows of `pitch` bytes).
int normalise_into(const tx_plan* p, const uint8_t* src, int64_t n, int64_t pitch, float* ring, int64_t pos,
                   unsigned long long* S, float2* muw, cudaStream_t st) {
  if (n <= 0) return TX_OK;
  TX_CUDA(cudaMemsetAsync(S, 0, (size_t)p->nchan * 16, st));
  const int ld = tf_load_form(src, p->nchan);
  if (p->layout == TX_LAYOUT_FT) {
    TX_CUDA(launch_pdl(k_chan_sums_ft, dim3((unsigned)((n + kSumBytes - 1) / kSumBytes), (unsigned)p->nchan),
                       dim3(kThreads), 0, st, src, n, pitch, S));
  } else {
    // about eight blocks per SM over the channel groups and times
    const int64_t groups = (p->nchan + 255) / 256, want = std::max<int64_t>(8 * p->dev.num_sms / groups, 1);
    const int chunk = (int)std::min<int64_t>(kSumBytes, std::max<int64_t>(64, ((n + want - 1) / want + 15) / 16 * 16));
    TX_CUDA(launch_pdl(k_chan_sums_tf, dim3((unsigned)((n + chunk - 1) / chunk), (unsigned)groups), dim3(kThreads), 0, st,
                       src, p->nchan, n, chunk, (int)(ld > 0), S));
  }
  TX_CUDA(launch_pdl(k_chan_weights, dim3((p->nchan + 127) / 128), dim3(128), 0, st, S, p->nchan, n, p->norm, muw));
  pos = mod(pos, p->R);
  const int64_t span = n + pos % 4;   // on the ring's 16-byte grid
  if (p->layout == TX_LAYOUT_FT)
    TX_CUDA(launch_pdl(k_norm_ingest_ft, dim3((unsigned)std::min<int64_t>((span + 4 * kThreads - 1) / (4 * kThreads), 64),
                                              (unsigned)p->nchan),
                       dim3(kThreads), 0, st, src, n, pitch, ring, p->R, pos, muw));
  else
    TX_CUDA(launch_pdl(k_norm_ingest_tf, dim3((unsigned)((span + 64 * kNormTiles - 1) / (64 * kNormTiles)),
                                              (unsigned)((p->nchan + 63) / 64)),
                       dim3(kThreads), 0, st, src, p->nchan, n, ring, p->R, pos, ld, muw));
  return TX_OK;
}

}  // namespace

int float_upload(tx_plan* p) {
  TX_CUDA(raise_smem_limit((const void*)k_stage1_f32, kF1Smem));
  TX_CUDA(upload_stage2_pipe32<float>(p));
  return TX_OK;
}

int float_wait_timeouts(int64_t* n) {
  int v = 0;
  TX_CUDA(cudaMemcpyFromSymbol(&v, g_tx_wait_timeouts, sizeof(int)));
  *n = v;
  return TX_OK;
}

int float_prime(const tx_plan* p, tx_beam* b, const uint8_t* d_tail, void* stream) {
  // the primed tail is normalised by its own statistics, as a block of L samples
  if (p->L <= 0) return TX_OK;
  const int64_t pitch = p->L;
  return normalise_into(p, d_tail, p->L, pitch, reinterpret_cast<float*>(b->ring), b->head - p->L,
                        reinterpret_cast<unsigned long long*>(b->chan),
                        reinterpret_cast<float2*>(b->chan + (size_t)p->nchan * 16), (cudaStream_t)stream);
}

int float_execute(const tx_plan* p, tx_beam* b, const uint8_t* d_block, void* d_out, int64_t* d_ncand,
                  void* d_workspace, void* stream, void* const* evp) {
  cudaStream_t st = (cudaStream_t)stream;
  const cudaEvent_t* ev = reinterpret_cast<const cudaEvent_t*>(evp);
  auto mark = [&](int i) -> int {
    if (ev) TX_CUDA(cudaEventRecord(ev[i], st));
    return TX_OK;
  };
  int rc;
  if ((rc = mark(0))) return rc;
  uint8_t* ws = static_cast<uint8_t*>(d_workspace);
  float* P = reinterpret_cast<float*>(ws + p->ws_P);
  const bool series = p->output == TX_OUT_SERIES;
  float* D = series ? static_cast<float*>(d_out) : reinterpret_cast<float*>(ws + p->ws_D);
  const int64_t Dp = series ? p->Td : p->Dp;
  double2* part = reinterpret_cast<double2*>(ws + p->ws_part);
  double2* ms = reinterpret_cast<double2*>(ws + p->ws_const);
  unsigned long long* S = reinterpret_cast<unsigned long long*>(ws + p->ws_hoff);
  float2* muw = reinterpret_cast<float2*>(ws + p->ws_hoff + (size_t)p->nchan * 16);
  float* ring = reinterpret_cast<float*>(b->ring);

  // Sec. 2.1 then Sec. 2.3 data flow: the block is normalised as it lands behind the tail
  const int64_t start = mod(b->head - p->L, p->R);
  if ((rc = normalise_into(p, d_block, p->T, p->T, ring, b->head, S, muw, st))) return rc;
  b->head = mod(b->head + p->T, p->R);
  if ((rc = mark(1))) return rc;

  // stage 1: the plan's items (sub-band, coarse DMs, time tile)
  F1Args f1{};
  f1.ring = ring;
  f1.items = p->dev.items_f;
  f1.chunks = p->dev.chunks_f;
  f1.tab = p->dev.tab_f;
  f1.abase = p->dev.abase;
  f1.P = P;
  f1.run = b->run;
  f1.R = p->R;
  f1.start = start;
  f1.Pp = p->Pp;
  f1.m = p->m;
  f1.nsub = p->nsub;
  f1.ndm = p->ndm;
  f1.nitems = (int32_t)p->items_f.size();
  f1.phase = p->phases_f == 1 ? 0 : (int32_t)(start & 3);
  f1.polls = first_wait_polls();
  TX_CUDA(launch_pdl(k_stage1_f32, dim3(std::min(f1.nitems, std::max(p->dev.num_sms, 1))), dim3(kF1Threads),
                     (size_t)kF1Smem, st, f1));
  if ((rc = mark(2))) return rc;

  // stage 2 with per-tile sums
  TX_CUDA(launch_stage2_pipe32<float>(p, P, D, Dp, part, b->run, st));
  if ((rc = mark(3))) return rc;

  if (!series) {
    k_stats_f32<<<(p->ndm + 127) / 128, 128, 0, st>>>(part, p->ntile2 * p->split32, p->ndm, p->T, p->stats == TX_STATS_RUNNING,
                                                      p->lambda, b->run, ms);
    TX_CUDA(cudaGetLastError());
    if ((rc = mark(4))) return rc;
    if (p->output == TX_OUT_CANDS) TX_CUDA(cudaMemsetAsync(d_ncand, 0, sizeof(int64_t), st));
    // units of the plan's boxcar length (the longest that still leaves a full
    // GPU several units per resident block)
    const int tile = p->box_tile;
    const int smem = (tile + p->wmax) * (int)sizeof(float2);
    // the most any plan needs (the attribute belongs to the current device)
    TX_CUDA(cudaFuncSetAttribute((const void*)k_boxcar_f32, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (4 * kBoxTile + kMaxWidth) * (int)sizeof(float2)));
    float* outf = static_cast<float*>(d_out);
    uint8_t* outw = p->output == TX_OUT_PLANE ? static_cast<uint8_t*>(d_out) + (size_t)p->ndm * p->T * 4 : nullptr;
    const int nt = (int)((p->T + tile - 1) / tile);   // units per DM
    k_boxcar_f32<<<p->ndm * nt, kThreads, smem, st>>>(
        D, Dp, p->T, tile, nt, ms, p->dev.widths, p->nw, p->wmax, p->output, p->gamma, outf, outw,
        static_cast<tx_cand*>(d_out), reinterpret_cast<unsigned long long*>(d_ncand), p->max_cands);
    TX_CUDA(cudaGetLastError());
  } else {
    if ((rc = mark(4))) return rc;
  }
  return mark(5);
}
