// Stage 2 (Sec. 2.3 sub-band step 3) from 32-bit intermediates, int32 or
// float32: D[d][t] = sum_s P[k(d)][s][t + d2[d][s]], with per-tile sums of D
// and D^2. Included by kernels.cu (int32) and floatpath.cu (float32).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "device.cuh"

namespace {

// Arguments of one launch. E is int32_t or float.
template <typename E>
struct Pipe32Args {
  const E* P;            // [nk][nsub][Pp]
  const int32_t* tab;    // per (coarse group, sub-band chunk): see tx_plan::tab2
  E* D;                  // [ndm][Dp]
  void* part;            // per (DM, tile, warp of the DM): longlong2 or double2 (sum D, sum D^2)
  double* run;           // the beam's running statistics, then its count of given-up waits
  int64_t Pp, Dp, Td, T;
  int32_t ndm, nsub, G, SC, SW;   // SC sub-bands per chunk, SW staged elements per sub-band
  int32_t ntile, nunits, nstage, split;
  uint32_t polls;
};

// Sums of D and D^2 over a warp's outputs, VW of them per lane (0 where there is
// none). Integers are exact. Floats: a lane's sum is carried as three float32 parts,
// what one part's add rounds off going into the next, the square as TwoProduct. The
// first two start at powers of two above any sum of the lane, so that an add's error
// takes two operations more (Dekker's FastTwoSum) instead of five; they are taken off
// again in double. The third's own rounding is below 2^-50 of the largest value, against
// up to 2^-43 for adding 32 values in double: nothing is lost to the double sums. (Two
// parts lose the second's rounding, up to 2^-43 of the sum, in the mean of equal values
// a hundred times the error of double sums, which a variance far below the squared mean
// magnifies.) A double add and multiply-add per output would cost 1.3 ms per 4096 x
// 65791 series at GB300's double rate.
template <int VW>
__device__ __forceinline__ longlong2 tile_sums(const int32_t (&x)[VW]) {
  long long s1 = 0;
  unsigned long long s2 = 0;
#pragma unroll
  for (int v = 0; v < VW; ++v) {
    s1 += x[v];
    s2 += (unsigned long long)((long long)x[v] * x[v]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
  }
  return make_longlong2(s1, (long long)s2);
}
struct Sum3 {
  float hi, mid, lo = 0.f;
  float hi0, mid0;
  // for up to 32 values below `top`, a power of two
  __device__ __forceinline__ explicit Sum3(float top) : hi(64.f * top), mid(64.f * 64.f * 0x1p-24f * top), hi0(hi), mid0(mid) {}
  static __device__ __forceinline__ float add_to(float& s, float x) {   // returns what the sum rounded off
    const float t = __fadd_rn(s, x), e = __fsub_rn(x, __fsub_rn(t, s));
    s = t;
    return e;
  }
  __device__ __forceinline__ void add_mid(float x) { lo = __fadd_rn(lo, add_to(mid, x)); }
  __device__ __forceinline__ void add(float x) { add_mid(add_to(hi, x)); }
  __device__ __forceinline__ double total() const {
    return ((double)hi - (double)hi0) + (((double)mid - (double)mid0) + (double)lo);
  }
};
template <int VW>
__device__ __forceinline__ double2 tile_sums(const float (&x)[VW]) {
  static_assert(VW <= 32, "Sum3 holds the sum of 32 values");
  float most = 0.f;
#pragma unroll
  for (int v = 0; v < VW; ++v) most = fmaxf(most, fabsf(x[v]));
  const float top = __uint_as_float((__float_as_uint(most) & 0x7F800000u) + 0x00800000u);   // the power of two above
  Sum3 s1(top), s2(top * top);
#pragma unroll
  for (int v = 0; v < VW; ++v) {
    s1.add(x[v]);
    const float p = __fmul_rn(x[v], x[v]);
    s2.add(p);
    s2.add_mid(__fmaf_rn(x[v], x[v], -p));
  }
  double a = s1.total(), b = s2.total();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  return make_double2(a, b);
}

// Persistent blocks walk units (coarse group k, tile of 32 VW split outputs)
// in sub-band chunks through `nstage` shared-memory stages. The last warp
// issues: it waits until every consumer has left a stage (mbarrier `empty`),
// then bulk-copies (TMA) the chunk's rows, one per lane, and its offset
// table; they complete `full`. The others sum: warp w takes part w % split of
// fine DM w / split (NDM = 2, groups of more than 16: also of the DM 16
// further), VW outputs per lane at stride 32, one conflict-free 32-bit load
// per sample-add whatever the delay. Copies and sums of different chunks
// overlap and nothing waits for the whole block.
// Bound: shared memory, 4 bytes per sample-add (39.1 TB/s measured: 1.77 ms
// for 17.3e9 sample-adds). Tiles of 1024 outputs keep the group's delay
// spread (up to about 440 samples on MeerKAT-L) a small part of what is
// staged, and 16 to 28 consumer warps of 8 to 32 independent sums keep the
// loads in flight. 4096 DMs x 64 sub-bands x 65791 outputs: float32 3.90 ->
// 2.02 ms, int32 11.99 -> 1.94 ms against one block per tile that staged its
// rows with 4-byte copies between block-wide barriers. Waits are bounded as
// in k_stage2_pipe.
template <typename E, int VW, int NDM>
__global__ void __launch_bounds__(VW * NDM >= 32 ? 544 : 928, 1)
k_stage2_pipe32(const Pipe32Args<E> a) {
  extern __shared__ __align__(16) uint8_t smem32[];
  pdl_wait();
  pdl_trigger();
  constexpr int kMaxStage = 3;
  __shared__ __align__(8) uint64_t full[kMaxStage], empty[kMaxStage];
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int NC = (int)(blockDim.x >> 5) - 1;                  // consumer warps
  const int SCq = (a.SC + 3) & ~3;
  const int tab_words = (a.G + 1) * SCq;
  const int stage_words = a.SC * a.SW + tab_words;
  const int nchunk = (a.nsub + a.SC - 1) / a.SC;
  const int tile_len = 32 * VW * a.split;
  uint32_t* smem = reinterpret_cast<uint32_t*>(smem32);
  if ((int)blockIdx.x >= a.nunits) return;
  if (threadIdx.x == 0) {
    for (int i = 0; i < a.nstage; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], NC);
    }
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  volatile int* abort = &abort_flag;
  auto give_up = [&]() {
    if (atomicExch(&abort_flag, 1) == 0) record_give_up(a);
  };

  if (warp == NC) {   // ---- the issuing warp
    int64_t q = 0;
    int st = 0;
    uint32_t ph = 1u;   // parity of the stage's previous use
    bool go = true;
    for (int u = blockIdx.x; u < a.nunits && go; u += gridDim.x) {
      const int k = u / a.ntile;
      const int64_t t0 = (int64_t)(u - k * a.ntile) * tile_len;
      for (int ch = 0; ch < nchunk; ++ch, ++q) {
        if (q >= a.nstage && !mbar_wait_warp(&empty[st], ph, a.polls, abort)) {
          give_up();
          go = false;
          break;
        }
        const int s0 = ch * a.SC, ns = min(a.SC, a.nsub - s0);
        const int32_t* tabk = a.tab + ((size_t)k * nchunk + ch) * tab_words;
        uint32_t* dst = smem + (size_t)st * stage_words;
        if (lane == 0) mbar_expect_tx(&full[st], ((uint32_t)ns * (uint32_t)a.SW + (uint32_t)tab_words) * 4u);
        __syncwarp();
        fence_proxy_async();
        for (int ss = lane; ss < ns; ss += 32) {
          const int64_t b = t0 + __ldg(tabk + (size_t)a.G * SCq + ss);
          bulk_g2s(dst + (size_t)ss * a.SW, a.P + ((size_t)k * a.nsub + s0 + ss) * a.Pp + b, (uint32_t)a.SW * 4u,
                   &full[st]);
        }
        if (lane == 0) bulk_g2s(dst + (size_t)a.SC * a.SW, tabk, (uint32_t)tab_words * 4u, &full[st]);
        if (++st == a.nstage) { st = 0; ph ^= 1u; }
      }
    }
    if (lane == 0) {
      // copies still in flight complete before the block's shared memory is released
      for (int64_t r = q > a.nstage ? q - a.nstage : 0; r < q; ++r)
        mbar_wait(&full[(int)(r % a.nstage)], (uint32_t)((r / a.nstage) & 1), kMbarPolls);
    }
    return;
  }

  // ---- consumers
  const int g = warp / a.split, part_i = warp - g * a.split;
  const int j0 = part_i * 32 * VW + lane;   // this lane's first output of the tile
  int st = 0;
  uint32_t ph = 0u;
  for (int u = blockIdx.x; u < a.nunits; u += gridDim.x) {
    const int k = u / a.ntile, tile = u - k * a.ntile;
    const int dfirst = k * a.G;
    const int nd = min(a.G, a.ndm - dfirst);
    E acc[NDM][VW];
#pragma unroll
    for (int n = 0; n < NDM; ++n)
#pragma unroll
      for (int v = 0; v < VW; ++v) acc[n][v] = (E)0;
    for (int ch = 0; ch < nchunk; ++ch) {
      if (!mbar_wait_warp(&full[st], ph, a.polls, abort)) {
        give_up();
        return;
      }
      const int ns = min(a.SC, a.nsub - ch * a.SC);
      const uint32_t* sw = smem + (size_t)st * stage_words;
      const E* rows = reinterpret_cast<const E*>(sw) + j0;
      const int32_t* tab = reinterpret_cast<const int32_t*>(sw + (size_t)a.SC * a.SW);
#pragma unroll
      for (int n = 0; n < NDM; ++n) {
        if (g + 16 * n >= nd) continue;
        const int32_t* t = tab + (g + 16 * n) * SCq;
#pragma unroll 2
        for (int ss = 0; ss < ns; ++ss) {
          const E* r = rows + ss * a.SW + t[ss];
#pragma unroll
          for (int v = 0; v < VW; ++v) {
            if constexpr (std::is_same<E, float>::value) acc[n][v] = __fadd_rn(acc[n][v], r[32 * v]);
            else acc[n][v] += r[32 * v];
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);
      if (++st == a.nstage) { st = 0; ph ^= 1u; }
    }
    // the unit's sums are complete: this warp's outputs and their sums
    const int64_t t0 = (int64_t)tile * tile_len + j0;
#pragma unroll
    for (int n = 0; n < NDM; ++n) {
      if (g + 16 * n >= nd) continue;
      const int d = dfirst + g + 16 * n;
      E* drow = a.D + (size_t)d * a.Dp;
#pragma unroll
      for (int v = 0; v < VW; ++v) {
        const int64_t t = t0 + 32 * v;
        if (t < a.Td) drow[t] = acc[n][v];
        if (t >= a.T) acc[n][v] = (E)0;
      }
      const auto tot = tile_sums(acc[n]);
      if (lane == 0)
        reinterpret_cast<std::remove_const_t<decltype(tot)>*>(a.part)[((size_t)d * a.ntile + tile) * a.split + part_i] =
            tot;
    }
  }
}

// The kernel for a plan's tile: VW outputs per lane (4 .. 32), one or two DMs per warp.
template <typename E>
using Pipe32Kernel = void (*)(const Pipe32Args<E>);
template <typename E>
Pipe32Kernel<E> pipe32_kernel(int vw, int ndm_per_warp) {
  if (ndm_per_warp == 2) return vw >= 16 ? k_stage2_pipe32<E, 16, 2> : k_stage2_pipe32<E, 8, 2>;
  switch (vw) {
    case 32: return k_stage2_pipe32<E, 32, 1>;
    case 16: return k_stage2_pipe32<E, 16, 1>;
    case 8: return k_stage2_pipe32<E, 8, 1>;
    default: return k_stage2_pipe32<E, 4, 1>;
  }
}

inline int pipe32_threads(const tx_plan* p) { return ((p->group > 16 ? 16 : p->group) * p->split32 + 1) * 32; }
inline int pipe32_smem(const tx_plan* p) { return (int)stage2_pipe32_smem(p->nstage32, p->nsub_chunk2, p->sw32, p->group); }
template <typename E>
Pipe32Kernel<E> pipe32_kernel(const tx_plan* p) {
  return pipe32_kernel<E>(p->tile32 / 32 / p->split32, p->group > 16 ? 2 : 1);
}

// Sets its shared memory limit and the blocks that share an SM: several for
// groups of few DMs (937 DMs in groups of 2, 2 sub-bands, 17507 outputs: 110 us
// with one block of 9 warps per SM, 33 us with the blocks that fit).
template <typename E>
cudaError_t upload_stage2_pipe32(tx_plan* p) {
  const Pipe32Kernel<E> k = pipe32_kernel<E>(p);
  cudaError_t e = raise_smem_limit((const void*)k, pipe32_smem(p));
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p->dev.s2_blocks_per_sm, k, pipe32_threads(p), pipe32_smem(p));
  return e;
}

// Launches the 32-bit stage 2 of plan p.
template <typename E>
cudaError_t launch_stage2_pipe32(const tx_plan* p, const E* P, E* D, int64_t Dp, void* part, double* run, cudaStream_t st) {
  Pipe32Args<E> a{};
  a.P = P;
  a.tab = p->dev.tab2;
  a.D = D;
  a.part = part;
  a.run = run;
  a.Pp = p->Pp;
  a.Dp = Dp;
  a.Td = p->Td;
  a.T = p->T;
  a.ndm = p->ndm;
  a.nsub = p->nsub;
  a.G = p->group;
  a.SC = p->nsub_chunk2;
  a.SW = p->sw32;
  a.ntile = p->ntile2;
  a.nunits = p->nk * p->ntile2;
  a.nstage = p->nstage32;
  a.split = p->split32;
  a.polls = first_wait_polls();
  const int grid = std::min(a.nunits, std::max(p->dev.num_sms, 1) * std::max(p->dev.s2_blocks_per_sm, 1));
  return launch_pdl(pipe32_kernel<E>(p), dim3(grid), dim3(pipe32_threads(p)), (size_t)pipe32_smem(p), st, a);
}

}  // namespace
