// Candidate clustering on the GPU (Sec. 2.5): DBSCAN on the DM-time plane,
// with DM converted to dispersion delay across the band (Eq. 1) so that both
// axes are in milliseconds.
//
//   core point      more than k other points at distance <= r
//   cluster         the core points connected by chains of core neighbours,
//                   with the non-core points within r of them
//   outlier         any other point
//
// The paper finds neighbours with a kd-tree (Sec. 2.5, O(log N) per query).
// Here the points, sorted by (DM index, time), are rows of times, and the
// neighbours of a point in another DM's row are those in one interval of times
// around it: its half length in samples depends on the two DMs only and comes
// from a table made with the clusterer (entries within rounding of a whole
// sample are marked, and the interval's end points then take the test in
// IEEE double, so that every decision is the double one). A query is a
// binary search per row, whatever the density.
//
// Steps (one stream, no host round trip):
//   1. canonical order: points sorted by (DM index, time) (radix sort), row starts;
//   2. neighbour counts, up to k + 1 -> core flags;
//   3. runs: a core point joins the core point before it in its row when that
//      is within r (head of each run by a max scan);
//   4. union-find over runs of different rows (lock-free: a root is linked under a
//      smaller root, so the final root of a cluster is its smallest canonical
//      index, which is the cluster's id): of the core points in an interval only
//      those are joined that no nearer one of them is already joined to, three
//      at most;
//   5. labels: a core point's root; a non-core point the smallest root among
//      its core neighbours, or -1;
//   6. per cluster: member count, DM and time extent, and the member of
//      highest S/N (ties: smallest canonical index), by integer atomics, one
//      set per warp and label;
//   7. compaction of the clusters in id order (exclusive scan).
// Every result is independent of thread order. What bounds it for a block's
// candidates is the chain of some twenty dependent launches (a third of it the
// radix sort's passes). Against visiting every pair within r through a grid of
// cells: 150 to 260 thousand candidates of six bright pulses (r = 4 ms, 2048
// DMs) 4.62 -> 0.29 ms; 52 thousand of a block whose pulses cover most of the
// plane (r = 8 ms) 79 -> 0.88 ms.
//
// Where more than kMaxRows DM trials lie within r of one, rows are the wrong
// index (a binary search for each, mostly empty); there a uniform grid of cells
// slightly larger than r takes steps 2 to 5: every neighbour lies in the 3 x 3
// cells around a point, and points sorted by cell make each cell row one
// contiguous range.
#include <cuda_runtime.h>

#include <cub/cub.cuh>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

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

struct tx_clusterer {
  int device = -1;
  double r = 0.0, cell = 0.0, tsamp_ms = 0.0;
  int32_t k = 0;
  int64_t cap = 0;
  int ndm = 0;
  double* table = nullptr;              // [ndm] delay per DM trial, ms
  unsigned long long *key_a = nullptr, *key_b = nullptr;
  int32_t *val_a = nullptr, *val_b = nullptr;
  int32_t* perm = nullptr;              // canonical index -> record index
  double *x = nullptr, *y = nullptr;    // canonical coordinates
  unsigned long long* ckey = nullptr;   // cell keys sorted
  int32_t* cidx = nullptr;              // canonical index of each sorted cell entry
  float *xs = nullptr, *ys = nullptr;   // per sorted entry: coordinates relative to its cell corner
  int32_t* core = nullptr;
  int32_t* parent = nullptr;
  int32_t* label = nullptr;
  int32_t* cnt = nullptr;
  unsigned long long* rep = nullptr;
  int32_t *dlo = nullptr, *dhi = nullptr, *tlo = nullptr, *thi = nullptr;
  int32_t* flag = nullptr;
  int32_t* pos = nullptr;
  void* temp = nullptr;
  size_t temp_bytes = 0;
  // rows: [ndm][nrow + 1] half interval between a DM and the i-th after it, in
  // samples, times 2, plus 1 when its end points need the double test; -1: out of
  // reach. Row starts [ndm + 1]. nrow < 0: the grid is used.
  int nrow = -1, sort_bits = 64;
  int32_t *reach = nullptr, *row = nullptr;
};

namespace {

constexpr int kThreads = 256;
constexpr int kMaxRows = 256;               // DM trials within r of one for the row index
constexpr int64_t kMaxReach = 1 << 24;      // entries of its table

__global__ void k_cl_canon(const tx_cand* __restrict__ c, int n, unsigned long long* key, int32_t* val) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  key[i] = ((unsigned long long)(uint32_t)c[i].dm_index << 32) | (uint32_t)c[i].t;
  val[i] = i;
}

__global__ void k_cl_coords(const tx_cand* __restrict__ c, const int32_t* __restrict__ perm, int n,
                            const double* __restrict__ table, double tsamp_ms, double cell, double* x, double* y,
                            unsigned long long* key, int32_t* val) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const tx_cand r = c[perm[j]];
  const double xv = table[r.dm_index];
  const double yv = __dmul_rn((double)r.t, tsamp_ms);
  x[j] = xv;
  y[j] = yv;
  const unsigned long long cx = (unsigned long long)floor(xv / cell), cy = (unsigned long long)floor(yv / cell);
  key[j] = (cx << 32) | cy;
  val[j] = j;
}

__device__ __forceinline__ int lower_bound(const unsigned long long* __restrict__ a, int n, unsigned long long v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Calls f(q) for every other point q within r of canonical point j, in cell
// order; f returns false to stop early. The test is
//   (x_q - x_j)^2 + (y_q - y_j)^2 <= r^2     in IEEE double,
// screened first in float on coordinates relative to the cell corner (errors
// below 1e-6 r^2): only pairs within 1e-5 r^2 of the radius take the double
// test, so every decision is the double one.
template <typename F>
__device__ __forceinline__ void for_neighbours(const tx_clusterer& C, int n, int j, F&& f) {
  const double xj = C.x[j], yj = C.y[j];
  const double r2 = __dmul_rn(C.r, C.r);
  const float r2f = (float)r2, lo2 = r2f * (1.0f - 1e-5f), hi2 = r2f * (1.0f + 1e-5f);
  const float cellf = (float)C.cell;
  const long long cx = (long long)floor(xj / C.cell), cy = (long long)floor(yj / C.cell);
  const float xjl = (float)(xj - (double)cx * C.cell), yjl = (float)(yj - (double)cy * C.cell);
  for (long long dx = -1; dx <= 1; ++dx) {
    if (cx + dx < 0) continue;
    const unsigned long long row = (unsigned long long)(cx + dx) << 32;
    const unsigned long long lo = row | (unsigned long long)(cy > 0 ? cy - 1 : 0);
    const unsigned long long hi = row | (unsigned long long)(cy + 1);
    for (int e = lower_bound(C.ckey, n, lo); e < n; ++e) {
      const unsigned long long key = C.ckey[e];
      if (key > hi) break;
      const float ddx = C.xs[e] - xjl + (float)dx * cellf;
      const float ddy = C.ys[e] - yjl + (float)((long long)(uint32_t)key - cy) * cellf;
      const float d2f = ddx * ddx + ddy * ddy;
      if (d2f > hi2) continue;
      const int q = C.cidx[e];
      if (q == j) continue;
      if (d2f >= lo2) {  // near the radius: decide in double
        const double gx = __dsub_rn(C.x[q], xj), gy = __dsub_rn(C.y[q], yj);
        if (!(__dadd_rn(__dmul_rn(gx, gx), __dmul_rn(gy, gy)) <= r2)) continue;
      }
      if (!f(q)) return;
    }
  }
}

// Cell-relative float coordinates of each sorted entry.
__global__ void k_cl_local(const tx_clusterer C, int n) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  const int q = C.cidx[e];
  const unsigned long long key = C.ckey[e];
  C.xs[e] = (float)(C.x[q] - (double)(key >> 32) * C.cell);
  C.ys[e] = (float)(C.y[q] - (double)(uint32_t)key * C.cell);
}

__global__ void k_cl_core(const tx_clusterer C, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  int cnt = 0;
  for_neighbours(C, n, j, [&](int) { return ++cnt <= C.k; });  // stop once core
  C.core[j] = cnt > C.k;
  C.parent[j] = j;
  C.cnt[j] = 0;
  C.rep[j] = 0ull;
  C.dlo[j] = INT32_MAX;
  C.dhi[j] = INT32_MIN;
  C.tlo[j] = INT32_MAX;
  C.thi[j] = INT32_MIN;
}

__device__ __forceinline__ int cl_find(int32_t* parent, int x) {
  volatile int32_t* p = parent;
  int px = p[x];
  while (px != x) {
    const int gp = p[px];
    if (gp != px) p[x] = gp;  // path halving: always an ancestor of x
    x = px;
    px = p[x];
  }
  return x;
}

// Joins the sets of p and q.
__device__ __forceinline__ void cl_unite(int32_t* parent, int p, int q) {
  int a = cl_find(parent, p);
  if (((volatile int32_t*)parent)[q] == a) return;  // already joined
  int b = cl_find(parent, q);
  while (a != b) {
    if (a < b) { const int t = a; a = b; b = t; }
    // link the larger root a under the smaller root b
    const int old = atomicCAS(parent + a, a, b);
    if (old == a) break;
    a = cl_find(parent, a);
    b = cl_find(parent, b);
  }
}

__global__ void k_cl_union(const tx_clusterer C, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n || !C.core[j]) return;
  for_neighbours(C, n, j, [&](int q) {
    if (q < j && C.core[q]) cl_unite(C.parent, j, q);  // each core pair once
    return true;
  });
}

__global__ void k_cl_label_core(const tx_clusterer C, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  C.label[j] = C.core[j] ? cl_find(C.parent, j) : -1;
}

__global__ void k_cl_label_border(const tx_clusterer C, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n || C.core[j]) return;
  int best = INT32_MAX;
  for_neighbours(C, n, j, [&](int q) {
    if (C.core[q]) best = min(best, C.label[q]);
    return true;
  });
  C.label[j] = best == INT32_MAX ? -1 : best;
}

__device__ __forceinline__ uint32_t ordered(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// A warp's points mostly share a label (they are neighbours in canonical
// order): one set of atomics per warp and label.
__global__ void k_cl_reduce(const tx_clusterer C, const tx_cand* __restrict__ c, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const int l = j < n ? C.label[j] : -1;
  tx_cand r{};
  if (l >= 0) r = c[C.perm[j]];
  const uint32_t snr = ordered(r.snr);
  for (unsigned todo = __ballot_sync(0xffffffffu, l >= 0); todo;) {
    const int lead = __ffs(todo) - 1;
    const int lab = __shfl_sync(0xffffffffu, l, lead);
    const bool in = l == lab;
    const unsigned grp = __ballot_sync(0xffffffffu, in);
    const uint32_t top = __reduce_max_sync(0xffffffffu, in ? snr : 0u);
    const uint32_t first = __reduce_max_sync(0xffffffffu, in && snr == top ? ~(uint32_t)j : 0u);
    const int dlo = __reduce_min_sync(0xffffffffu, in ? r.dm_index : INT32_MAX);
    const int dhi = __reduce_max_sync(0xffffffffu, in ? r.dm_index : INT32_MIN);
    const int tlo = __reduce_min_sync(0xffffffffu, in ? r.t : INT32_MAX);
    const int thi = __reduce_max_sync(0xffffffffu, in ? r.t : INT32_MIN);
    if (lane == lead) {
      atomicAdd(C.cnt + lab, __popc(grp));
      atomicMax(C.rep + lab, ((unsigned long long)top << 32) | first);
      atomicMin(C.dlo + lab, dlo);
      atomicMax(C.dhi + lab, dhi);
      atomicMin(C.tlo + lab, tlo);
      atomicMax(C.thi + lab, thi);
    }
    todo &= ~grp;
  }
}

__global__ void k_cl_flag(const tx_clusterer C, int n, int32_t* flag) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  flag[j] = C.core[j] && C.label[j] == j;
}

__global__ void k_cl_emit(const tx_clusterer C, const tx_cand* __restrict__ c, int n, tx_cluster* out,
                          int64_t* nclusters, int32_t* labels_out, int32_t* order_out) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  if (labels_out) labels_out[j] = C.label[j];
  if (order_out) order_out[j] = C.perm[j];
  if (j == n - 1) *nclusters = (int64_t)C.pos[j] + C.flag[j];
  if (!C.flag[j]) return;
  const unsigned long long rk = C.rep[j];
  const int best = (int)(~(uint32_t)(rk & 0xFFFFFFFFull));
  const tx_cand r = c[C.perm[best]];
  tx_cluster o;
  o.id = j;
  o.dm_index = r.dm_index;
  o.t = r.t;
  o.w_index = r.w_index;
  o.snr = r.snr;
  o.members = C.cnt[j];
  o.dm_lo = C.dlo[j];
  o.dm_hi = C.dhi[j];
  o.t_lo = C.tlo[j];
  o.t_hi = C.thi[j];
  out[C.pos[j]] = o;
}
// ---- rows -------------------------------------------------------------------
// The DM index of a canonical key (one that is no trial of the plan: ndm, a row
// without neighbours).
__device__ __forceinline__ int cl_dm(const tx_clusterer& C, unsigned long long key) {
  return (int)min((unsigned long long)C.ndm, key >> 32);
}

// row[d] = first canonical index of DM d or later, d <= ndm; and what the
// other steps start from.
__global__ void k_cl_rows(const tx_clusterer C, const unsigned long long* __restrict__ key, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int d = cl_dm(C, key[j]), before = j ? cl_dm(C, key[j - 1]) : -1;
  for (int e = before + 1; e <= d; ++e) C.row[e] = j;
  if (j == n - 1)
    for (int e = d + 1; e <= C.ndm; ++e) C.row[e] = n;
  C.cnt[j] = 0;
  C.rep[j] = 0ull;
  C.dlo[j] = INT32_MAX;
  C.dhi[j] = INT32_MIN;
  C.tlo[j] = INT32_MAX;
  C.thi[j] = INT32_MIN;
}

// (x_q - x_p)^2 + (y_q - y_p)^2 <= r^2 in IEEE double.
__device__ __forceinline__ bool cl_near(const tx_clusterer& C, int dp, uint32_t tp, int dq, uint32_t tq) {
  const double gx = __dsub_rn(C.table[dq], C.table[dp]);
  const double gy = __dsub_rn(__dmul_rn((double)(int32_t)tq, C.tsamp_ms), __dmul_rn((double)(int32_t)tp, C.tsamp_ms));
  return __dadd_rn(__dmul_rn(gx, gx), __dmul_rn(gy, gy)) <= __dmul_rn(C.r, C.r);
}

// Calls f(lo, hi) for the times of row dq within r of point (d, t) (reach: the
// table's entry for the two DMs), as intervals of the order of the keys, in which
// negative times come last: one, or two where the times around t change sign. The
// row is not empty. f returns false to stop.
template <typename F>
__device__ __forceinline__ bool cl_interval(const tx_clusterer& C, const unsigned long long* __restrict__ key, int d,
                                            uint32_t tu, int dq, int reach, F&& f) {
  const int t = (int)tu, h = reach >> 1;
  int lo = t >= INT32_MIN + h ? t - h : INT32_MIN;
  int hi = t <= INT32_MAX - h ? t + h : INT32_MAX;
  if (reach & 1) {
    const bool in_lo = t < INT32_MIN + h || cl_near(C, d, tu, dq, (uint32_t)lo);
    const bool in_hi = t > INT32_MAX - h || cl_near(C, d, tu, dq, (uint32_t)hi);
    if (h == 0 && !(in_lo && in_hi)) return true;   // none
    lo += !in_lo;
    hi -= !in_hi;
  }
  uint32_t a = (uint32_t)(hi >= 0 ? max(lo, 0) : lo), b = (uint32_t)hi;
#pragma unroll 1   // f once in the code
  while (f(a, b)) {
    if (lo >= 0 || a == (uint32_t)lo || (int)(uint32_t)key[C.row[dq + 1] - 1] >= 0) return true;   // (none negative)
    a = (uint32_t)lo;
    b = 0xFFFFFFFFu;
  }
  return false;
}

// First entry of [b, e) whose time is at least t.
__device__ __forceinline__ int cl_search(const unsigned long long* __restrict__ key, int b, int e, uint32_t t) {
  while (b < e) {
    const int mid = (b + e) >> 1;
    if ((uint32_t)key[mid] < t) b = mid + 1; else e = mid;
  }
  return b;
}

// Calls f(dq, reach) for the non-empty rows within r of row d, the point's own
// first, then outwards; f returns false to stop.
template <typename F>
__device__ __forceinline__ void cl_rows(const tx_clusterer& C, int d, bool before, F&& f) {
  const int w = C.nrow + 1;
  if (d >= C.ndm) return;
  if (!f(d, __ldg(C.reach + (size_t)d * w))) return;
  bool up = true, down = before;
  for (int i = 1; i <= C.nrow && (up || down); ++i) {
    if (up) {
      const int q = d + i;
      const int h = q < C.ndm ? __ldg(C.reach + (size_t)d * w + i) : -1;
      if (h < 0) up = false;
      else if (C.row[q] < C.row[q + 1] && !f(q, h)) return;
    }
    if (down) {
      const int q = d - i;
      const int h = q >= 0 ? __ldg(C.reach + (size_t)q * w + i) : -1;
      if (h < 0) down = false;
      else if (C.row[q] < C.row[q + 1] && !f(q, h)) return;
    }
  }
}

__global__ void k_cl_row_core(const tx_clusterer C, const unsigned long long* __restrict__ key, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int d = cl_dm(C, key[j]);
  const uint32_t t = (uint32_t)key[j];
  long long cnt = -1;   // the point itself is counted
  cl_rows(C, d, true, [&](int q, int reach) {
    return cl_interval(C, key, d, t, q, reach, [&](uint32_t lo, uint32_t hi) {
      const int e = C.row[q + 1];
      int p;
      if (q == d && lo <= t && t <= hi) {   // up to k + 1 to the left of the point, then on to the right
        p = j;
        while (p > C.row[d] && (uint32_t)key[p - 1] >= lo && j - p <= C.k) --p;
      } else {
        p = cl_search(key, C.row[q], e, lo);
      }
      for (; p < e && (uint32_t)key[p] <= hi && cnt <= C.k; ++p) ++cnt;
      return cnt <= C.k;
    });
  });
  C.core[j] = cnt > C.k;
}

// val[j] = j for the head of a run of core points, else 0: a core point whose
// row's core point before it is out of reach. Times of one sign make a run.
__global__ void k_cl_row_heads(const tx_clusterer C, const unsigned long long* __restrict__ key, int n, int32_t* val) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  int v = 0;
  if (C.core[j]) {
    const int d = cl_dm(C, key[j]);
    const uint32_t t = (uint32_t)key[j];
    v = j;
    cl_interval(C, key, d, t, d, __ldg(C.reach + (size_t)d * (C.nrow + 1)), [&](uint32_t lo, uint32_t hi) {
      if (t < lo || t > hi) return true;
      for (int p = j - 1; p >= C.row[d] && (uint32_t)key[p] >= lo; --p)
        if (C.core[p]) { v = 0; break; }
      return false;
    });
  }
  val[j] = v;
}

// Calls f(p) for core points p of the interval [lo, hi] of row q: the first, and
// after each the first that is out of its reach (those in its reach are joined
// to it already, own0 being the row's reach in itself).
template <typename F>
__device__ __forceinline__ void cl_cores(const tx_clusterer& C, const unsigned long long* __restrict__ key, int q,
                                         uint32_t lo, uint32_t hi, F&& f) {
  const int e = C.row[q + 1];
  const int own = __ldg(C.reach + (size_t)q * (C.nrow + 1));
  const uint32_t step = (uint32_t)(own >> 1) - ((own & 1) && own > 1 ? 1u : 0u);
  int p = cl_search(key, C.row[q], e, lo);
  while (true) {
    while (p < e && (uint32_t)key[p] <= hi && !C.core[p]) ++p;
    if (p >= e || (uint32_t)key[p] > hi) return;
    f(p);
    if (step >= hi - (uint32_t)key[p]) return;
    const uint32_t nt = (uint32_t)key[p] + step;   // the last time certainly in p's reach
    p = cl_search(key, p + 1, e, nt + 1);
  }
}

__global__ void k_cl_row_union(const tx_clusterer C, const unsigned long long* __restrict__ key, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n || !C.core[j]) return;
  const int d = cl_dm(C, key[j]);
  const uint32_t t = (uint32_t)key[j];
  cl_rows(C, d, false, [&](int q, int reach) {   // each pair of rows once: later rows only
    if (q == d && ((int)t < 0 || (int)t > (reach >> 1))) return true;   // (of the own row: negative times from the others)
    return cl_interval(C, key, d, t, q, reach, [&](uint32_t lo, uint32_t hi) {
      if (q != d || (int)lo < 0) cl_cores(C, key, q, lo, hi, [&](int p) { cl_unite(C.parent, j, p); });
      return true;
    });
  });
}

// Labels of the core points, and the flags of the clusters' first points.
__global__ void k_cl_row_label(const tx_clusterer C, int n, int32_t* flag) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int l = C.core[j] ? cl_find(C.parent, j) : -1;
  C.label[j] = l;
  flag[j] = l == j;
}

// parent = the head of a core point's run (val after the max scan)
__global__ void k_cl_row_parent(const tx_clusterer C, const int32_t* __restrict__ val, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) C.parent[j] = C.core[j] ? val[j] : j;
}

__global__ void k_cl_row_border(const tx_clusterer C, const unsigned long long* __restrict__ key, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n || C.core[j]) return;
  const int d = cl_dm(C, key[j]);
  const uint32_t t = (uint32_t)key[j];
  int best = INT32_MAX;
  cl_rows(C, d, true, [&](int q, int reach) {
    return cl_interval(C, key, d, t, q, reach, [&](uint32_t lo, uint32_t hi) {
      cl_cores(C, key, q, lo, hi, [&](int p) { best = min(best, C.label[p]); });
      return true;
    });
  });
  C.label[j] = best == INT32_MAX ? -1 : best;
}

struct Larger {
  __device__ __forceinline__ int32_t operator()(int32_t a, int32_t b) const { return a > b ? a : b; }
};

template <typename T>
int dalloc(T** p, int64_t n) {
  TX_CUDA(cudaMalloc((void**)p, (size_t)std::max<int64_t>(n, 1) * sizeof(T)));
  return TX_OK;
}

// Steps 2 to 5 on rows; canonical keys in key_b, flags to fl.
int run_rows(tx_clusterer* C, int ni, int32_t* fl, cudaStream_t st) {
  const int grid = (ni + kThreads - 1) / kThreads;
  const unsigned long long* key = C->key_b;
  k_cl_rows<<<grid, kThreads, 0, st>>>(*C, key, ni);
  k_cl_row_core<<<grid, kThreads, 0, st>>>(*C, key, ni);
  k_cl_row_heads<<<grid, kThreads, 0, st>>>(*C, key, ni, C->flag);
  TX_CUDA(cudaGetLastError());
  size_t tb = C->temp_bytes;
  TX_CUDA(cub::DeviceScan::InclusiveScan(C->temp, tb, C->flag, C->pos, Larger{}, ni, st));
  k_cl_row_parent<<<grid, kThreads, 0, st>>>(*C, C->pos, ni);
  k_cl_row_union<<<grid, kThreads, 0, st>>>(*C, key, ni);
  k_cl_row_label<<<grid, kThreads, 0, st>>>(*C, ni, fl);
  k_cl_row_border<<<grid, kThreads, 0, st>>>(*C, key, ni);
  TX_CUDA(cudaGetLastError());
  return TX_OK;
}

// Steps 2 to 5 on a grid of cells.
int run_grid(tx_clusterer* C, const tx_cand* d_cands, int ni, int32_t* fl, cudaStream_t st) {
  const int grid = (ni + kThreads - 1) / kThreads;
  // coordinates and cells
  k_cl_coords<<<grid, kThreads, 0, st>>>(d_cands, C->perm, ni, C->table, C->tsamp_ms, C->cell, C->x, C->y,
                                         C->key_a, C->val_a);
  TX_CUDA(cudaGetLastError());
  unsigned long long* ck = C->key_b;       // canonical keys are no longer needed
  int32_t* ci = reinterpret_cast<int32_t*>(C->flag);
  size_t tb = C->temp_bytes;
  TX_CUDA(cub::DeviceRadixSort::SortPairs(C->temp, tb, C->key_a, ck, C->val_a, ci, ni, 0, 64, st));
  C->ckey = ck;
  C->cidx = ci;
  k_cl_local<<<grid, kThreads, 0, st>>>(*C, ni);
  // core flags, union-find, labels
  k_cl_core<<<grid, kThreads, 0, st>>>(*C, ni);
  k_cl_union<<<grid, kThreads, 0, st>>>(*C, ni);
  k_cl_label_core<<<grid, kThreads, 0, st>>>(*C, ni);
  k_cl_label_border<<<grid, kThreads, 0, st>>>(*C, ni);
  k_cl_flag<<<grid, kThreads, 0, st>>>(*C, ni, fl);
  TX_CUDA(cudaGetLastError());
  return TX_OK;
}

}  // namespace

extern "C" {

int32_t tx_clusterer_create(const tx_plan* p, double radius_ms, int32_t k, int64_t max_points, tx_clusterer** out) {
  if (!p || !out) { set_error("null argument"); return TX_ERR_INVALID_ARG; }
  *out = nullptr;
  if (!(radius_ms > 0.0) || k < 0 || max_points < 1 || max_points >= INT32_MAX) {
    set_error("need radius_ms > 0, k >= 0 and 1 <= max_points < 2^31");
    return TX_ERR_INVALID_ARG;
  }
  tx_clusterer* C = new (std::nothrow) tx_clusterer();
  if (!C) { set_error("out of host memory"); return TX_ERR_OOM; }
  cudaGetDevice(&C->device);
  C->r = radius_ms;
  C->cell = radius_ms * (1.0 + 1e-9);  // a neighbour within r is never two cells away
  C->tsamp_ms = p->tsamp * 1e3;
  C->k = k;
  C->cap = max_points;
  C->ndm = p->ndm;
  const int64_t n = max_points;
  int rc = TX_OK;
  while (C->sort_bits > 33 && ((int64_t)1 << (C->sort_bits - 33)) >= p->ndm) --C->sort_bits;   // 32 + bits of a DM index
  // rows: the half intervals, unless too many DMs lie within r of one
  std::vector<int32_t> reach;
  {
    const std::vector<double>& x = p->delay_ms;
    const volatile double r2 = radius_ms * radius_ms;
    int most = 0;
    for (int d = 0, e = 0; d < p->ndm && most <= kMaxRows; ++d) {
      for (e = std::max(e, d); e + 1 < p->ndm; ++e) {
        const double gx = x[e + 1] - x[d];
        const volatile double g2 = gx * gx;
        if (!(g2 <= r2)) break;
      }
      most = std::max(most, e - d);
    }
    if (most <= kMaxRows && (int64_t)p->ndm * (most + 1) <= kMaxReach && radius_ms / C->tsamp_ms < 5e8) {
      C->nrow = most;
      try {
        reach.assign((size_t)p->ndm * (most + 1), -1);
      } catch (const std::bad_alloc&) {
        set_error("out of host memory");
        tx_clusterer_destroy(C);
        return TX_ERR_OOM;
      }
      for (int d = 0; d < p->ndm; ++d)
        for (int i = 0; i <= most && d + i < p->ndm; ++i) {
          const double gx = x[d + i] - x[d];
          const volatile double g2 = gx * gx;
          if (!(g2 <= r2)) break;
          // r^2 - gx^2 in samples squared; the test's own rounding moves it by far less than `slack`
          const double q = std::max(0.0, (r2 - g2) / (C->tsamp_ms * C->tsamp_ms)), h = std::floor(std::sqrt(q));
          const double slack = 1e-5 * (h + 1.0) + 1e-12 * (r2 / (C->tsamp_ms * C->tsamp_ms));
          const bool next = (h + 1.0) * (h + 1.0) - q <= slack;
          reach[(size_t)d * (most + 1) + i] = 2 * (int32_t)(next ? h + 1.0 : h) + (next || q - h * h <= slack ? 1 : 0);
        }
    }
  }
  if (!rc) rc = dalloc(&C->table, p->ndm);
  if (!rc) rc = dalloc(&C->row, (int64_t)p->ndm + 1);
  if (!rc) rc = dalloc(&C->reach, (int64_t)reach.size());
  if (!rc) rc = dalloc(&C->key_a, n);
  if (!rc) rc = dalloc(&C->key_b, n);
  if (!rc) rc = dalloc(&C->val_a, n);
  if (!rc) rc = dalloc(&C->val_b, n);
  if (!rc) rc = dalloc(&C->x, n);
  if (!rc) rc = dalloc(&C->y, n);
  if (!rc) rc = dalloc(&C->core, n);
  if (!rc) rc = dalloc(&C->parent, n);
  if (!rc) rc = dalloc(&C->label, n);
  if (!rc) rc = dalloc(&C->cnt, n);
  if (!rc) rc = dalloc(&C->rep, n);
  if (!rc) rc = dalloc(&C->dlo, n);
  if (!rc) rc = dalloc(&C->dhi, n);
  if (!rc) rc = dalloc(&C->tlo, n);
  if (!rc) rc = dalloc(&C->thi, n);
  if (!rc) rc = dalloc(&C->flag, n);
  if (!rc) rc = dalloc(&C->pos, n);
  if (!rc) rc = dalloc(&C->xs, n);
  if (!rc) rc = dalloc(&C->ys, n);
  if (!rc && cudaMemcpy(C->table, p->delay_ms.data(), p->delay_ms.size() * sizeof(double),
                        cudaMemcpyHostToDevice) != cudaSuccess) {
    set_error("delay table upload failed");
    rc = TX_ERR_CUDA;
  }
  if (!rc && !reach.empty() &&
      cudaMemcpy(C->reach, reach.data(), reach.size() * sizeof(int32_t), cudaMemcpyHostToDevice) != cudaSuccess) {
    set_error("interval table upload failed");
    rc = TX_ERR_CUDA;
  }
  if (!rc) {
    size_t a = 0, b = 0, c = 0;
    cub::DeviceRadixSort::SortPairs(nullptr, a, C->key_a, C->key_b, C->val_a, C->val_b, (int)n);
    cub::DeviceScan::ExclusiveSum(nullptr, b, C->flag, C->pos, (int)n);
    cub::DeviceScan::InclusiveScan(nullptr, c, C->flag, C->pos, Larger{}, (int)n);
    C->temp_bytes = std::max(a, std::max(b, c));
    if (cudaMalloc(&C->temp, std::max<size_t>(C->temp_bytes, 16)) != cudaSuccess) {
      set_error("clusterer scratch allocation failed");
      rc = TX_ERR_OOM;
    }
  }
  if (rc) { tx_clusterer_destroy(C); return rc; }
  *out = C;
  return TX_OK;
}

int32_t tx_cluster_run(tx_clusterer* C, const tx_cand* d_cands, int64_t n, tx_cluster* d_out, int64_t* d_nclusters,
                       int32_t* d_labels, int32_t* d_order, void* stream) {
  if (!C || (!d_cands && n > 0) || !d_out || !d_nclusters) { set_error("null argument"); return TX_ERR_INVALID_ARG; }
  if (n < 0 || n > C->cap) { set_error("%lld points, capacity %lld", (long long)n, (long long)C->cap); return TX_ERR_INVALID_ARG; }
  cudaStream_t st = (cudaStream_t)stream;
  if (n == 0) {
    TX_CUDA(cudaMemsetAsync(d_nclusters, 0, sizeof(int64_t), st));
    return TX_OK;
  }
  const int ni = (int)n;
  const int grid = (ni + kThreads - 1) / kThreads;
  size_t tb = C->temp_bytes;
  // 1. canonical order
  k_cl_canon<<<grid, kThreads, 0, st>>>(d_cands, ni, C->key_a, C->val_a);
  TX_CUDA(cudaGetLastError());
  TX_CUDA(cub::DeviceRadixSort::SortPairs(C->temp, tb, C->key_a, C->key_b, C->val_a, C->val_b, ni, 0, C->sort_bits, st));
  C->perm = C->val_b;
  int32_t* fl = C->val_a;   // flags of the clusters' first points
  if (C->nrow >= 0) {
    if (const int rc = run_rows(C, ni, fl, st)) return rc;
  } else if (const int rc = run_grid(C, d_cands, ni, fl, st)) {
    return rc;
  }
  // 6. per-cluster reductions
  k_cl_reduce<<<grid, kThreads, 0, st>>>(*C, d_cands, ni);
  // 7. clusters in id order
  tx_clusterer Cf = *C;
  Cf.flag = fl;
  tb = C->temp_bytes;
  TX_CUDA(cub::DeviceScan::ExclusiveSum(C->temp, tb, fl, C->pos, ni, st));
  k_cl_emit<<<grid, kThreads, 0, st>>>(Cf, d_cands, ni, d_out, d_nclusters, d_labels, d_order);
  TX_CUDA(cudaGetLastError());
  return TX_OK;
}

void tx_clusterer_destroy(tx_clusterer* C) {
  if (!C) return;
  int prev = 0;
  cudaGetDevice(&prev);
  if (C->device >= 0) cudaSetDevice(C->device);
  for (void* q : {(void*)C->table, (void*)C->key_a, (void*)C->key_b, (void*)C->val_a, (void*)C->val_b, (void*)C->x,
                  (void*)C->y, (void*)C->core, (void*)C->parent, (void*)C->label, (void*)C->cnt, (void*)C->rep,
                  (void*)C->dlo, (void*)C->dhi, (void*)C->tlo, (void*)C->thi, (void*)C->flag, (void*)C->pos,
                  (void*)C->xs, (void*)C->ys, (void*)C->reach, (void*)C->row, C->temp})
    cudaFree(q);
  cudaSetDevice(prev);
  delete C;
}

}  // extern "C"
