// Truncated series of Lemma 2.3 on the GPU: h^(L) = sum_{i=0}^{L} P^i D^{-1} b_st
// and beta^(L) = ||h||^2 - (1^T h)^2 / n (Eq. tr-beta-exp-Liu), for batches of
// queries (the deterministic quantity the paper's PUSH computes).
//
// Arithmetic: GB300 issues FP64 at about 2 lane operations per SM per clock,
// against 128 for FP32, and an FP64 step was bound by that pipe.  x, y and h
// are therefore held as double-float pairs (hi + lo, two FP32 values with
// |lo| <= ulp(hi)/2, a 48-bit significand), added and multiplied with exact
// error-free transformations (TwoSum, and TwoProd by fused multiply-add), each
// a handful of FP32 operations; the final reduction to beta is FP64.
//
// C = 4, 8, 16 or 32 queries per pass (the fewest columns that hold what is left
// of a group of equal L), one warp lane per query column and 32 / C rows per
// warp.  x, y and h are n x C row-major, so gathering x over a node's neighbours
// reads whole sectors (C = 32: two lines a row).  Iteration i forms x_{i+1} =
// P x_i with (P x)_v = (sum_{u in N(v)} x_u) * (1/d_v), neighbours read from
// col_idx (4 bytes per entry); every second iteration adds x_i and x_{i+1} to h,
// which halves the traffic of h.
//
// Rows of at most 64 entries take one warp's lanes and add in CSR order; longer
// rows are cut into segments of 64 or of about the root of their degree, whose
// partial sums are added in segment order by the warp that finishes the row's
// last one.  An addition of pairs is a chain of about 50 clocks, so a row's
// length is its latency: with 1024-entry segments, and the heavy rows in two
// launches after the light ones, a step on a 10^5-node power-law graph waited
// 155 us for its two hubs where all other rows took 20.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <string>
#include <vector>

#include "pw_device.cuh"
#include "pw_internal.h"

namespace pw {

constexpr int kSeriesCols = 32;       // most queries per pass
constexpr int32_t kSeriesRow = 64;    // rows with more entries are cut into segments
constexpr int64_t kSeriesSegment = 64;  // entries of a segment, or about the root of the row's if more
constexpr int kSeriesThreads = 256;
// Scratch up to this size stays with the graph until it is freed (cudaMalloc and
// cudaFree wait for the device); larger is allocated and freed by each call.
constexpr size_t kSeriesKeptBytes = (size_t)256 << 20;

// ---- double-float arithmetic (value = hi + lo) -----------------------------
// TwoSum (Knuth): s + e == a + b exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Sum of two pairs; both parts by TwoSum, then renormalised (relative error
// about 2^-46 of the result).
__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
  float s1, e1, s2, e2;
  two_sum(a.x, b.x, s1, e1);
  two_sum(a.y, b.y, s2, e2);
  e1 = __fadd_rn(e1, s2);
  float h = __fadd_rn(s1, e1);
  e1 = __fsub_rn(e1, __fsub_rn(h, s1));
  e1 = __fadd_rn(e1, e2);
  const float hi = __fadd_rn(h, e1);
  return make_float2(hi, __fsub_rn(e1, __fsub_rn(hi, h)));
}

// Product of two pairs; TwoProd of the high parts by fused multiply-add.
__device__ __forceinline__ float2 df_mul(float2 a, float2 b) {
  const float p = __fmul_rn(a.x, b.x);
  float e = __fmaf_rn(a.x, b.x, -p);
  e = __fmaf_rn(a.x, b.y, e);
  e = __fmaf_rn(a.y, b.x, e);
  const float hi = __fadd_rn(p, e);
  return make_float2(hi, __fsub_rn(e, __fsub_rn(hi, p)));
}

__device__ __forceinline__ float2 df_from_double(double v) {
  const float hi = __double2float_rn(v);
  return make_float2(hi, __double2float_rn(v - (double)hi));
}

// Start vectors D^{-1} (e_s - e_t) of a pass, into zeroed x.
__global__ void series_seed_kernel(float2* __restrict__ x, const int2* __restrict__ st, int ncols, int cols,
                                   const int4* __restrict__ node) {
  const int c = threadIdx.x;
  if (c >= ncols) return;
  const int s = st[c].x, t = st[c].y;
  if (s == t) return;
  x[(size_t)s * cols + c] = df_from_double(1.0 / (double)node[s].z);
  x[(size_t)t * cols + c] = df_from_double(-1.0 / (double)node[t].z);
}

// 1/d_v as a pair, once per call.
__global__ void series_inv_degree_kernel(const int4* __restrict__ node, float2* __restrict__ inv, uint32_t n) {
  for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
    inv[v] = df_from_double(1.0 / (double)__ldg(&node[v].z));
}

struct SeriesArgs {
  const float2* x;
  float2* y;
  float2* h;
  const int32_t* col;
  const int4* node;
  const float2* inv;
  const int2* rows;       // {e_begin, entries} of each row, entries -1 for heavy rows; [n] = {0, -1}
  const int4* segs;       // {heavy row, e_begin, e_end, partial slot}
  const int4* heavy;      // {row, first partial slot, partial count, -}
  float2* partial;        // nseg x C
  unsigned int* arrived;  // per heavy row: segments done in this step (wraps to 0)
  uint32_t n;
  int32_t nseg;
};

// Sum of many pairs: the high parts by TwoSum, their errors and the low parts
// in FP32 sums of their own, normalised now and then (fold) and at the end.  8
// operations a pair and a chain of one addition, against df_add's 20 and a
// chain of 12; the roundings are 2^-25 of sums of terms 2^-25 of the first, as
// df_add's are.
struct PairSum {
  float hi = 0.f, err = 0.f, low = 0.f;
  __device__ __forceinline__ void add(float2 v) {
    float s, e;
    two_sum(hi, v.x, s, e);
    hi = s;
    err = __fadd_rn(err, e);
    low = __fadd_rn(low, v.y);
  }
  __device__ __forceinline__ void fold() {
    const float t = __fadd_rn(err, low);
    float s;
    two_sum(hi, t, s, low);
    hi = s;
    err = 0.f;
  }
  __device__ __forceinline__ float2 value() {
    fold();
    return make_float2(hi, low);
  }
};

// The first C neighbour ids of a row of len entries, one per lane of its part;
// past the row's end the index of the zero row after x's last, n.
template <int C>
__device__ __forceinline__ uint32_t series_ids(const int32_t* __restrict__ col, int32_t e0, int32_t len, uint32_t sub,
                                               uint32_t n) {
  return (int32_t)sub < len ? (uint32_t)__ldg(col + e0 + (int32_t)sub) : n;
}

// Sum of x_u (column = lane mod C) over the entries [e0, e0 + len) of one row,
// in CSR order, folded after every 8 entries whatever C, so that a query's bits do
// not depend on the pass's width (a fold past a row's end changes nothing); every
// lane of the warp calls, 32 / C rows at once.  `mine`: the
// row's first ids (series_ids), the next C come with one coalesced load; up to 8
// row loads are in flight.  Rows shorter than the warp's longest add the zero
// row, which leaves a sum unchanged.  An entry costs a shuffle, an address, a
// load and 8 additions; a predicate and a zero for each had cost as much again.
template <int C>
__device__ __forceinline__ float2 series_row_sum(const float2* __restrict__ x, const int32_t* __restrict__ col,
                                                 uint32_t mine, int32_t e0, int32_t len, uint32_t sub, uint32_t n) {
  PairSum acc;
  const int32_t longest = C == 32 ? len : __reduce_max_sync(0xffffffffu, len);
  const float2* mycol = x + sub;
  for (int32_t b = 0; b < longest; b += C) {
    const int32_t lim = longest - b < C ? longest - b : C;  // the same in the whole warp
    const uint32_t next = b + C < longest ? series_ids<C>(col, e0 + b + C, len - b - C, sub, n) : n;
    for (int32_t j = 0; j < lim; j += 8) {
      const int32_t rem = lim - j;
      float2 v[8];
      auto load = [&](int q) {
        const uint32_t u = __shfl_sync(0xffffffffu, mine, j + q, C);
        v[q] = __ldg(mycol + (size_t)u * C);
      };
      auto two = [&](int q) {
        acc.add(v[q]);
        acc.add(v[q + 1]);
      };
      load(0);
      load(1);
      if (rem > 2) load(2), load(3);
      if (C > 4 && rem > 4) load(4), load(5);
      if (C > 4 && rem > 6) load(6), load(7);
      two(0);
      if (rem > 2) two(2);
      if (C > 4 && rem > 4) two(4);
      if (C > 4 && rem > 6) two(6);
      if (rem > 8) acc.fold();
    }
    // leaving here is up to 2 % faster than not, but 0.6 % slower with a row per warp
    if (C < 32 && b + C >= longest) break;
    if (C == 32 ? b + C < longest : C > 4 || (b & 4)) acc.fold();
    mine = next;
  }
  return acc.value();
}

// One iteration over all rows.  ACC: 0 leaves h, 1 adds x_i and then x_{i+1},
// 2 starts h as their sum.  The segments of heavy rows come first.
// Bound by issue (two thirds of the slots) and the latency of a row's loads on
// graphs in L2, by L2 and HBM bandwidth beyond; 5 blocks per SM (48 registers)
// against 6 (40): 258 and 277 us a step on a 1000^2 grid.  Microseconds a step,
// with a warp per row of up to 1,024 entries and always 32 columns -> now:
// 10^5-node power-law graph, 32 / 16 / 4 columns 168 -> 44 / 175 -> 28 / 168 ->
// 17; R-MAT 2^20, 32 / 8 columns 1,498 -> 1,110 / 1,499 -> 318; 2000^2 grid, 32
// columns 1,540 -> 1,037.
template <int C, int ACC>
__global__ void __launch_bounds__(kSeriesThreads, 5) series_step_kernel(SeriesArgs A) {
  constexpr uint32_t kRows = 32 / C;
  const uint32_t lane = threadIdx.x & 31u, sub = lane % C, part = lane / C;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  const uint32_t seg_groups = ((uint32_t)A.nseg + kRows - 1) / kRows;
  const uint32_t row_groups = (A.n + kRows - 1) / kRows;
  const float2 zero = make_float2(0.f, 0.f);
  auto finish = [&](size_t at, float2 sum, float2 inv, float2 x, float2 h) {
    const float2 y = df_mul(sum, inv);
    A.y[at] = y;
    if (ACC == 1) {
      PairSum sum_h{h.x, 0.f, h.y};
      sum_h.add(x);
      sum_h.add(y);
      A.h[at] = sum_h.value();
    }
    if (ACC == 2) A.h[at] = df_add(x, y);
  };
  uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  for (; g < seg_groups; g += warps) {
    const uint32_t i = g * kRows + part;
    const bool valid = i < (uint32_t)A.nseg;
    const int4 sg = valid ? __ldg(A.segs + i) : make_int4(0, 0, 0, 0);
    const int32_t len = sg.z - sg.y;
    const float2 sum = series_row_sum<C>(A.x, A.col, series_ids<C>(A.col, sg.y, len, sub, A.n), sg.y, len, sub, A.n);
    if (valid) __stcg(A.partial + (size_t)sg.w * C + sub, sum);
    __threadfence();
    __syncwarp();
    const int4 hr = valid ? __ldg(A.heavy + sg.x) : make_int4(0, 0, 0, 0);
    unsigned int before = 0;
    if (valid && sub == 0) before = atomicInc(A.arrived + sg.x, (unsigned int)hr.z - 1u);
    before = __shfl_sync(0xffffffffu, before, part * C);
    if (valid && before + 1u == (unsigned int)hr.z) {
      __threadfence();
      const size_t at = (size_t)(uint32_t)hr.x * C + sub;
      const float2 inv = __ldg(A.inv + hr.x), x = ACC ? A.x[at] : zero, h = ACC == 1 ? A.h[at] : zero;
      PairSum acc;
      const float2* p = A.partial + (size_t)hr.y * C + sub;
      int32_t k = 0;
      for (; k + 8 <= hr.z; k += 8) {
        float2 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = __ldcg(p + (size_t)(k + q) * C);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc.add(v[q]);
        acc.fold();
      }
      for (; k < hr.z; ++k) acc.add(__ldcg(p + (size_t)k * C));
      finish(at, acc.value(), inv, x, h);
    }
    __syncwarp();
  }
  // A row's own values are loaded before its neighbours', its first neighbour
  // ids one row ahead and its record two rows ahead.
  g -= seg_groups;
  uint32_t v = g * kRows + part;
  const uint32_t step = warps * kRows;
  auto record = [&](uint32_t u) { return __ldg(A.rows + (u < A.n ? u : A.n)); };
  int2 r0 = record(v), r1 = record(v + step);
  uint32_t ids = series_ids<C>(A.col, r0.x, r0.y, sub, A.n);
  size_t at = (size_t)v * C + sub;
  for (; g < row_groups; g += warps) {
    const bool light = r0.y >= 0;
    const float2 inv = light ? __ldg(A.inv + v) : zero;
    const float2 x = ACC && light ? A.x[at] : zero, h = ACC == 1 && light ? A.h[at] : zero;
    const uint32_t ids_next = series_ids<C>(A.col, r1.x, r1.y, sub, A.n);
    const int2 r2 = record(v + 2 * step);
    const float2 sum = series_row_sum<C>(A.x, A.col, ids, r0.x, light ? r0.y : 0, sub, A.n);
    if (light) finish(at, sum, inv, x, h);
    r0 = r1;
    r1 = r2;
    ids = ids_next;
    v += step;
    at += (size_t)step * C;
  }
}

// beta of each column: sums of h^2 and of h over the nodes in FP64, then
// sq - tot^2 / n.  h is A.h (use_h) plus A.x (use_x: the last x when its step
// did not add it).  Every block sums its rows and a tree its threads; the last
// block adds the blocks' sums, each in a fixed order.
template <int C>
__global__ void __launch_bounds__(8 * C) series_reduce_kernel(const float2* __restrict__ h,
                                                                       const float2* __restrict__ x, int use_h,
                                                                       int use_x, uint32_t n, int ncols,
                                                                       double* block_sums, unsigned int* arrived,
                                                                       double* __restrict__ out) {
  constexpr uint32_t kRows = 8;  // rows at once per block, for every C: the order of the sums is the same
  __shared__ double ssq[kRows * C], stot[kRows * C];
  __shared__ bool last;
  const uint32_t tid = threadIdx.x, c = tid % C;
  double sq = 0.0, tot = 0.0;
  for (uint64_t v = (uint64_t)blockIdx.x * kRows + tid / C; v < n; v += (uint64_t)gridDim.x * kRows) {
    const size_t at = (size_t)v * C + c;
    float2 p = use_h ? h[at] : make_float2(0.f, 0.f);
    if (use_x) p = use_h ? df_add(p, x[at]) : x[at];
    const double d = (double)p.x + (double)p.y;
    sq += d * d;
    tot += d;
  }
  auto tree = [&]() {
    ssq[tid] = sq;
    stot[tid] = tot;
    __syncthreads();
    for (uint32_t w = kRows * C / 2; w >= (uint32_t)C; w >>= 1) {
      if (tid < w) {
        ssq[tid] += ssq[tid + w];
        stot[tid] += stot[tid + w];
      }
      __syncthreads();
    }
  };
  tree();
  if (tid < (uint32_t)C) {
    __stcg(block_sums + ((size_t)blockIdx.x * C + c) * 2, ssq[tid]);
    __stcg(block_sums + ((size_t)blockIdx.x * C + c) * 2 + 1, stot[tid]);
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicInc(arrived, gridDim.x - 1u) + 1u == gridDim.x;
  __syncthreads();
  if (!last) return;
  __threadfence();
  sq = tot = 0.0;
  for (uint32_t b = tid / C; b < gridDim.x; b += kRows) {
    sq += __ldcg(block_sums + ((size_t)b * C + c) * 2);
    tot += __ldcg(block_sums + ((size_t)b * C + c) * 2 + 1);
  }
  tree();
  if ((int)tid < ncols) out[tid] = ssq[tid] - stot[tid] * stot[tid] / (double)n;
}

using SeriesStepFn = void (*)(SeriesArgs);
template <int C>
static SeriesStepFn series_step_fn(int acc) {
  return acc == 0 ? series_step_kernel<C, 0> : (acc == 1 ? series_step_kernel<C, 1> : series_step_kernel<C, 2>);
}

// One pass of `ncols` <= C queries of equal L, enqueued on `stream`; returns
// the number of kernels.  x_buf and y_buf alternate.
template <int C>
static int series_pass(SeriesArgs A, float2* x_buf, float2* y_buf, const int2* st, int ncols, int32_t L, int grid,
                       int reduce_grid, double* block_sums, unsigned int* reduce_arrived, double* out,
                       cudaStream_t stream) {
  // x_0 and the zero rows after the last
  cudaMemsetAsync(x_buf, 0, sizeof(float2) * ((size_t)A.n + 1) * C, stream);
  cudaMemsetAsync(y_buf + (size_t)A.n * C, 0, sizeof(float2) * C, stream);
  series_seed_kernel<<<1, kSeriesCols, 0, stream>>>(x_buf, st, ncols, C, A.node);
  float2 *x = x_buf, *y = y_buf;
  for (int32_t i = 0; i < L; ++i) {
    A.x = x;
    A.y = y;
    series_step_fn<C>((i & 1) ? 0 : (i == 0 ? 2 : 1))<<<grid, kSeriesThreads, 0, stream>>>(A);
    std::swap(x, y);
  }
  series_reduce_kernel<C><<<reduce_grid, 8 * C, 0, stream>>>(A.h, x, L > 0, (L & 1) == 0, A.n, ncols,
                                                                      block_sums, reduce_arrived, out);
  return L + 2;
}

// Rows and heavy rows' segments, laid out once per graph (they depend on its degrees only).
static pw_status series_plan(pw_graph* g) {
  SeriesPlan& P = g->series;
  if (P.ready) return PW_OK;
  std::vector<int4> segs, heavy;
  std::vector<int2> rows((size_t)g->n + 1, make_int2(0, -1));
  int64_t start = 0;
  int32_t slot = 0;
  for (int64_t v = 0; v < g->n; ++v) {
    const int32_t d = g->deg[(size_t)v];
    if (d > kSeriesRow) {
      int64_t size = kSeriesSegment;
      while (size * size < d) size *= 2;
      const int32_t first = slot;
      for (int64_t e = start; e < start + d; e += size)
        segs.push_back(make_int4((int)heavy.size(), (int)e, (int)std::min<int64_t>(e + size, start + d), slot++));
      heavy.push_back(make_int4((int)v, first, slot - first, 0));
    } else {
      rows[(size_t)v] = make_int2((int)start, d);
    }
    start += d;
  }
  pw_status st;
  if ((st = ensure_buffer(P.rows, sizeof(int2) * rows.size())) != PW_OK) return st;
  if ((st = ensure_buffer(P.segs, sizeof(int4) * segs.size())) != PW_OK) return st;
  if ((st = ensure_buffer(P.heavy, sizeof(int4) * heavy.size())) != PW_OK) return st;
  if ((st = ensure_buffer(P.arrived, sizeof(unsigned int) * (heavy.size() + 1))) != PW_OK) return st;
  PW_CUDA_TRY(cudaMemcpyAsync(P.rows.ptr, rows.data(), sizeof(int2) * rows.size(), cudaMemcpyHostToDevice, g->stream));
  PW_CUDA_TRY(cudaMemcpyAsync(P.segs.ptr, segs.data(), sizeof(int4) * segs.size(), cudaMemcpyHostToDevice, g->stream));
  PW_CUDA_TRY(cudaMemcpyAsync(P.heavy.ptr, heavy.data(), sizeof(int4) * heavy.size(), cudaMemcpyHostToDevice,
                              g->stream));
  PW_CUDA_TRY(cudaMemsetAsync(P.arrived.ptr, 0, sizeof(unsigned int) * (heavy.size() + 1), g->stream));
  PW_CUDA_TRY(cudaStreamSynchronize(g->stream));
  P.nseg = (int32_t)segs.size();
  P.nheavy = (int32_t)heavy.size();
  P.ready = true;
  return PW_OK;
}

}  // namespace pw

using namespace pw;

extern "C" pw_status pw_series_batch(pw_graph* g, int64_t count, const int64_t* s, const int64_t* t, const int32_t* L,
                                     double* beta_L) {
  if (!g) return set_error(PW_ERR_ARG, "graph is NULL");
  if (count < 0) return set_error(PW_ERR_ARG, "count < 0");
  if (count == 0) return PW_OK;
  if (!s || !t || !L || !beta_L) return set_error(PW_ERR_ARG, "NULL array");
  for (int64_t i = 0; i < count; ++i)
    if (s[i] < 0 || s[i] >= g->n || t[i] < 0 || t[i] >= g->n || L[i] < 0)
      return set_error(PW_ERR_ARG, "query " + std::to_string(i) + ": node id out of range or L < 0");
  std::lock_guard<std::mutex> guard(g->lock);
  PW_CUDA_TRY(cudaSetDevice(g->device));
  const size_t n = (size_t)g->n;
  cudaStream_t stream = g->stream;
  pw_status st = series_plan(g);
  if (st != PW_OK) return st;
  SeriesPlan& P = g->series;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, series_step_kernel<32, 1>, kSeriesThreads, 0) != cudaSuccess ||
      occ < 1)
    occ = 1;
  // blocks of a step: as many warps as the pass has rows and segments to hand out
  auto step_blocks = [&](int cols) {
    const int64_t groups = (int64_t)(n * (size_t)cols + 31) / 32 + ((int64_t)P.nseg * cols + 31) / 32;
    return (groups * 32 + kSeriesThreads - 1) / kSeriesThreads;
  };
  const int64_t resident = (int64_t)g->sm_count * occ;
  // queries with the same L share a pass: group by L in input order
  std::vector<int64_t> order((size_t)count);
  for (int64_t i = 0; i < count; ++i) order[(size_t)i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int64_t a, int64_t b) { return L[a] < L[b]; });
  // Where the resident warps have a row each at most, a step is short beside its launch,
  // and a group of several passes is captured once as a CUDA graph of 32 columns and
  // replayed, its last pass, which may hold fewer, too.  Launched each -> replayed: 1,000
  // queries at L = 200 on 200 nodes 32.5 -> 20.1 ms, 33 at L = 2000 20.5 -> 15.4, 64 at L =
  // 200 on 2,000 nodes 3.96 -> 3.44.  The capture costs what some 32 replayed steps save
  // (two passes on 200 nodes: 0.40 ms either way at L = 32, 0.17 -> 0.21 at L = 8); from
  // 64 on it pays (three passes at L = 32 0.55 -> 0.53).
  struct Pass {
    size_t begin;
    int ncols, cols;
    bool replay;
  };
  std::vector<Pass> passes;
  int most = 0;  // columns of the widest pass
  for (size_t pos = 0, group_end = 0; pos < order.size();) {
    bool replay = pos < group_end && passes.back().replay;
    if (pos == group_end) {
      while (group_end < order.size() && L[order[group_end]] == L[order[pos]]) ++group_end;
      const int64_t again = (int64_t)((group_end - pos - 1) / (size_t)kSeriesCols);  // passes after the first
      replay = again * L[order[pos]] >= 64 && step_blocks(kSeriesCols) <= resident;
    }
    const int ncols = (int)std::min(group_end - pos, (size_t)kSeriesCols);
    const int cols = replay || ncols > 16 ? 32 : (ncols <= 4 ? 4 : (ncols <= 8 ? 8 : 16));
    passes.push_back({pos, ncols, cols, replay});
    most = std::max(most, cols);
    pos += (size_t)ncols;
  }
  const int reduce_grid = g->sm_count * 4;
  // x, y, h, 1/d, partial sums, the reduction's block sums, (s, t) and results, and those of a replayed pass
  auto align = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t b_vec = align(sizeof(float2) * (n + 1) * (size_t)most), b_inv = align(sizeof(float2) * n);
  const size_t b_part = align(sizeof(float2) * (size_t)most * (size_t)P.nseg);
  const size_t b_sums = align(sizeof(double) * 2 * (size_t)most * (size_t)reduce_grid);
  const size_t b_st = align(sizeof(int2) * (size_t)count), b_out = align(sizeof(double) * (size_t)count);
  const size_t b_pass_st = align(sizeof(int2) * kSeriesCols), b_pass_out = align(sizeof(double) * kSeriesCols);
  const size_t bytes = 3 * b_vec + b_inv + b_part + b_sums + b_st + b_out + b_pass_st + b_pass_out;
  DeviceBuffer own;
  DeviceBuffer& buf = bytes <= kSeriesKeptBytes ? P.scratch : own;
  if ((st = ensure_buffer(buf, bytes)) != PW_OK) return st;
  char* at = (char*)buf.ptr;
  auto take = [&](size_t b) {
    char* p = at;
    at += b;
    return p;
  };
  float2* xb = (float2*)take(b_vec);
  float2* yb = (float2*)take(b_vec);
  SeriesArgs A;
  memset(&A, 0, sizeof A);
  A.h = (float2*)take(b_vec);
  float2* inv = (float2*)take(b_inv);
  A.partial = (float2*)take(b_part);
  double* sums = (double*)take(b_sums);
  int2* d_st = (int2*)take(b_st);
  double* d_out = (double*)take(b_out);
  int2* pass_st = (int2*)take(b_pass_st);
  double* pass_out = (double*)take(b_pass_out);
  A.inv = inv;
  A.col = g->d_col;
  A.node = g->d_node;
  A.rows = (const int2*)P.rows.ptr;
  A.segs = (const int4*)P.segs.ptr;
  A.heavy = (const int4*)P.heavy.ptr;
  A.arrived = (unsigned int*)P.arrived.ptr;
  unsigned int* reduce_arrived = A.arrived + P.nheavy;
  A.n = (uint32_t)n;
  A.nseg = P.nseg;
  std::vector<int2> h_st((size_t)count);
  for (size_t j = 0; j < order.size(); ++j) h_st[j] = make_int2((int)s[order[j]], (int)t[order[j]]);
  cudaError_t e = cudaMemcpyAsync(d_st, h_st.data(), sizeof(int2) * (size_t)count, cudaMemcpyHostToDevice, stream);
  series_inv_degree_kernel<<<g->sm_count * occ, kSeriesThreads, 0, stream>>>(g->d_node, inv, (uint32_t)n);
  count_launch();
  cudaGraphExec_t exec = nullptr;
  int32_t exec_L = -1;
  int exec_kernels = 0;
  for (const Pass& p : passes) {
    if (e != cudaSuccess) break;
    const int32_t Lc = L[order[p.begin]];
    const int grid = (int)std::min(resident, step_blocks(p.cols));
    const auto pass = p.cols == 4 ? series_pass<4> : (p.cols == 8 ? series_pass<8> : (p.cols == 16 ? series_pass<16> : series_pass<32>));
    if (p.replay && exec_L != Lc) {
      if (exec) {
        e = cudaStreamSynchronize(stream);
        cudaGraphExecDestroy(exec);
        exec = nullptr;
      }
      cudaGraph_t graph = nullptr;
      if (e == cudaSuccess) e = cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal);
      if (e != cudaSuccess) break;
      exec_kernels = pass(A, xb, yb, pass_st, kSeriesCols, Lc, grid, reduce_grid, sums, reduce_arrived, pass_out, stream);
      const cudaError_t e_launch = cudaGetLastError();
      e = cudaStreamEndCapture(stream, &graph);  // always ends the capture
      if (e == cudaSuccess) e = e_launch;
      if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
      if (graph) cudaGraphDestroy(graph);
      if (e != cudaSuccess) break;
      exec_L = Lc;
    }
    cudaEvent_t ev = nullptr;
    prof_begin(g, stream, &ev);
    if (p.replay) {  // the group's first pass is full, so every column has a query
      e = cudaMemcpyAsync(pass_st, d_st + p.begin, sizeof(int2) * (size_t)p.ncols, cudaMemcpyDeviceToDevice, stream);
      if (e == cudaSuccess) e = cudaGraphLaunch(exec, stream);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_out + p.begin, pass_out, sizeof(double) * (size_t)p.ncols, cudaMemcpyDeviceToDevice, stream);
      count_launches(exec_kernels);
    } else {
      count_launches(pass(A, xb, yb, d_st + p.begin, p.ncols, Lc, grid, reduce_grid, sums, reduce_arrived,
                          d_out + p.begin, stream));
    }
    prof_end(g, stream, ev, 3);
    if (g->prof.enabled) g->prof.series_steps += (uint64_t)Lc + 1;
    const cudaError_t e_last = cudaGetLastError();
    if (e == cudaSuccess) e = e_last;
  }
  std::vector<double> res((size_t)count);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(res.data(), d_out, sizeof(double) * (size_t)count, cudaMemcpyDeviceToHost, stream);
  const cudaError_t e_sync = cudaStreamSynchronize(stream);  // also before `own` and the host arrays go
  if (e == cudaSuccess) e = e_sync;
  if (exec) cudaGraphExecDestroy(exec);
  free_buffer(own);
  if (e != cudaSuccess) return cuda_error(e, "series");
  for (size_t j = 0; j < order.size(); ++j) {
    const int64_t i = order[j];
    beta_L[i] = s[i] == t[i] ? 0.0 : res[j];
  }
  return PW_OK;
}
