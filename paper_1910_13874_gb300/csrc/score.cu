// Scoring a given group (problem (i) of Section 2.1, Algorithm 1): one group by the
// paper's two-state hit/miss recurrences, many groups as columns of one SpMM.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "device_util.cuh"
#include "internal.h"
#include "run.h"

namespace gw {
namespace {

// X0[v] = (h_0(v), m_0(v)) = (1_S(v), 1_{V\S}(v)), times s on a weighted graph
template <typename T>
__global__ void init_two_state(T* __restrict__ X, const uint32_t* __restrict__ mask, int32_t n, const T* __restrict__ rs) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const bool inS = (mask[v >> 5] >> (v & 31)) & 1u;
    const T x = rs ? rs[v] : T(1);
    X[2 * static_cast<size_t>(v)] = inS ? x : T(0);
    X[2 * static_cast<size_t>(v) + 1] = inS ? T(0) : x;
  }
}

// Batched scoring of a directed graph, first-visit form. Column j of a block is m_0 = 1_{V \ S_j}.
// Isolated rows (r >= n_active) hold 0: the sweeps never write them and nothing gathers them,
// so they read as the (zero) first-visit counts of such vertices. (The autotuner starts from it too.)
__global__ void init_batch(float* __restrict__ X, int32_t n, int32_t n_active, int32_t cols, int32_t active) {
  const size_t total = static_cast<size_t>(n) * cols;
  const size_t live = static_cast<size_t>(n_active) * cols;
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < total; i += size_t(gridDim.x) * blockDim.x)
    X[i] = (i < live && static_cast<int32_t>(i % cols) < active) ? 1.0f : 0.0f;
}

__global__ void zero_members(float* __restrict__ X, int32_t cols, const int32_t* __restrict__ mrow,
                             const int32_t* __restrict__ mcol, int32_t count) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) X[static_cast<size_t>(mrow[i]) * cols + mcol[i]] = 0.0f;
}

// After sweep p: Y_p(s, j) = alpha (A m_{p-1})(s) is alpha^p F_p(s), the weighted p-walks whose
// first visit to S_j is their last vertex s. It meets every walk continuing from s:
// acc += alpha^p F_p(s) * K_{L-p}(s), K_q(s) = sum_{r<=q} t_r(s). Then m_p(s) = 0.
__global__ void batch_member_epilogue(float* __restrict__ Y, int32_t cols, const int32_t* __restrict__ mrow,
                                      const int32_t* __restrict__ mcol, double* __restrict__ acc, int32_t count,
                                      const double* __restrict__ ttab, int32_t n, int32_t q) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int32_t s = mrow[i];
  float* y = Y + static_cast<size_t>(s) * cols + mcol[i];
  const double f = static_cast<double>(*y);
  double K = 0.0;
  for (int32_t r = 0; r <= q; ++r) K += ttab[static_cast<size_t>(r) * n + s];
  acc[i] += f * K;
  *y = 0.0f;
}

// acc starts with the p = 0 term: every walk that starts at s (length 1..L) hits S_j at s.
__global__ void batch_member_init(const int32_t* __restrict__ mrow, double* __restrict__ acc, int32_t count,
                                  const double* __restrict__ ttab, int32_t n, int32_t L) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int32_t s = mrow[i];
  double K = 0.0;
  for (int32_t r = 1; r <= L; ++r) K += ttab[static_cast<size_t>(r) * n + s];
  acc[i] = K;
}

// score_j = sum over the members of group j, in member order.
__global__ void batch_group_sum(const double* __restrict__ acc, const int32_t* __restrict__ goff, int32_t groups,
                                double* __restrict__ out) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= groups) return;
  double s = 0.0;
  for (int32_t i = goff[j]; i < goff[j + 1]; ++i) s += acc[i];
  out[j] = s;
}

// ---------------------------------------------------------------- half-length batches (undirected)
// Column j of a block is the hit vector h_t(v) = the walks of length t that end at v and visit S_j:
// h_t = alpha A h_{t-1}, and on S_j every walk that ends there, h_t(s) = t_t(s), a row of the
// walk-total table. A walk of length H + a hits S_j in its half of length a or else in the other:
//   sum_v [ h_a(v) t_H(v) + (t_a(v) - h_a(v)) h_H(v) ],
// so ceil(L/2) vectors (the first from counts) and one pass over them replace L sweeps: 512 groups on
// a Barabasi-Albert graph of n = 10^6 (L = 9, blocks of 16 columns) took 41.2 ms with the first-visit
// sweeps of the full length.

// What a vertex contributes beside the hit vectors, as pairs (hi, lo) from the FP64 table: with x the
// stored vectors (s h on a weighted graph, i = 1 / s; s = 1 else) its term of the score is
//   i K(x) + i t_H V(x) + (s P - V(x)) i^2 x_H,   P = t_1 + .. + t_{L-H}.
struct BatchRow {
  Pair t, p;  // i t_H and s P
};
struct BatchScale {
  Pair i, i2;
};
__global__ void batch_totals(const double* __restrict__ T, int64_t n, int32_t n_active, int32_t L, int32_t H,
                             const double* __restrict__ rs, BatchRow* __restrict__ row, BatchScale* __restrict__ scale) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n_active; v += gridDim.x * blockDim.x) {
    const double inv = rs ? 1.0 / rs[v] : 1.0;
    double p = 0.0;
    for (int32_t a = 1; a <= L - H; ++a) p += T[static_cast<size_t>(a) * n + v];
    row[v] = BatchRow{to_pair(T[static_cast<size_t>(H) * n + v] * inv * inv), to_pair(p)};
    if (rs) scale[v] = BatchScale{to_pair(inv), to_pair(inv * inv)};
  }
}

// |N(v) cap S_j| outside the groups, as whole numbers in X's cells, and its rows' bits in nz.
// batch_count_scale makes them h_1 = alpha |N(v) cap S_j|, rounded once (adding alpha up in FP32 drifts with
// the count: 2.7e-4 of the score on a star of 100,000 leaves). With blockIdx.y = 0 a warp takes a member and
// up to kScatterRow entries of its row; the other slices of the grid (where rows are longer) look through
// up to 32 members at a time for the rest of hubs' rows, which they share.
constexpr int kScatterRow = 256;
__global__ void batch_scatter(int32_t* __restrict__ X, int32_t cols, const int32_t* __restrict__ mrow,
                              const int32_t* __restrict__ mcol, int32_t count, const int32_t* __restrict__ rp,
                              const int32_t* __restrict__ ci, uint32_t* __restrict__ nz) {
  const int lane = threadIdx.x & 31;
  const int32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, warps = (gridDim.x * blockDim.x) >> 5;
  auto add = [&](int64_t e, int32_t c) {
    const int32_t u = ci[e];
    atomicAdd(X + static_cast<size_t>(u) * cols + c, 1);
    if (!((nz[u >> 5] >> (u & 31)) & 1u)) atomicOr(nz + (u >> 5), 1u << (u & 31));
  };
  if (blockIdx.y == 0) {
    for (int32_t i = warp; i < count; i += warps) {
      const int32_t s = mrow[i], c = mcol[i];
      const int64_t e0 = rp[s], e1 = min(static_cast<int64_t>(rp[s + 1]), e0 + kScatterRow);
#pragma unroll 4
      for (int64_t e = e0 + lane; e < e1; e += 32) add(e, c);
    }
    return;
  }
  const int slice = static_cast<int>(blockIdx.y) - 1, slices = static_cast<int>(gridDim.y) - 1;
  const int per = max(1, min(32, (count + warps - 1) / warps));  // few members: each its own warps
  for (int64_t i0 = per * static_cast<int64_t>(warp); i0 < count; i0 += per * static_cast<int64_t>(warps)) {
    const bool some = lane < per && i0 + lane < count;
    const int32_t mine = some ? mrow[i0 + lane] : -1, col = some ? mcol[i0 + lane] : 0;
    const bool hub = mine >= 0 && rp[mine + 1] - rp[mine] > kScatterRow;
    for (unsigned m = __ballot_sync(kFullMask, hub); m; m &= m - 1) {
      const int32_t s = __shfl_sync(kFullMask, mine, __ffs(m) - 1), c = __shfl_sync(kFullMask, col, __ffs(m) - 1);
      const int64_t e1 = rp[s + 1];
#pragma unroll 4
      for (int64_t e = static_cast<int64_t>(rp[s]) + kScatterRow + slice * 32 + lane; e < e1; e += 32 * slices) add(e, c);
    }
  }
}

// The counts of the rows in nz (the others are 0 in either form) to alpha times them. A warp takes the 32
// rows of a word, four columns per lane; most words are 0 and skipped.
__global__ void batch_count_scale(float* __restrict__ X, int32_t cols, int32_t n_active, float alpha,
                                  const uint32_t* __restrict__ nz) {
  const int lane = threadIdx.x & 31, per = cols / 4, rows = 32 / per;  // rows at a time
  const int32_t words = (n_active + 31) / 32, warps = (gridDim.x * blockDim.x) >> 5;
  for (int32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < words; w += warps) {
    const uint32_t bits = nz[w];
    if (bits == 0) continue;
    for (int r0 = 0; r0 < 32; r0 += rows) {
      const int r = r0 + lane / per;
      if (!(bits >> r & 1u)) continue;
      const size_t q = (static_cast<size_t>(w) * 32 + r) * per + lane % per;
      const int4 k = reinterpret_cast<const int4*>(X)[q];
      reinterpret_cast<float4*>(X)[q] = make_float4(alpha * static_cast<float>(k.x), alpha * static_cast<float>(k.y),
                                                    alpha * static_cast<float>(k.z), alpha * static_cast<float>(k.w));
    }
  }
}

// h_t on the groups' own rows: a row of the table (as stored: times s on a weighted graph).
__global__ void batch_own(float* __restrict__ X, int32_t cols, const int32_t* __restrict__ mrow,
                          const int32_t* __restrict__ mcol, int32_t count, const double* __restrict__ row,
                          int32_t n_active, uint32_t* __restrict__ nz) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count || mrow[i] >= n_active) return;
  if (nz) atomicOr(nz + (mrow[i] >> 5), 1u << (mrow[i] & 31));
  X[static_cast<size_t>(mrow[i]) * cols + mcol[i]] = static_cast<float>(row[mrow[i]]);
}

// The stored vectors of a block: x_t sits at slot (t - 1) % slots; V holds the sum of those already
// folded (walk lengths 1..folded). Five slots hold the walks of L <= 10; two where five would outgrow
// kWideBytes or the device.
constexpr int kBatchRing = 5;
struct BatchVecs {
  const float* ring;
  int64_t stride;
  int slots;
  float* V;  // hi and lo parts, `stride` elements each
  int32_t folded, H;
};

// V (+)= x_{folded+1} .. x_{folded+slots-1}.
__global__ void batch_fold(const BatchVecs b, int64_t quads) {
  float4* hi = reinterpret_cast<float4*>(b.V);
  float4* lo = reinterpret_cast<float4*>(b.V + b.stride);
  for (int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < quads;
       q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    Pair a[4] = {};
    if (b.folded > 0) {
      const float4 h = hi[q], l = lo[q];
      a[0] = Pair{h.x, l.x}, a[1] = Pair{h.y, l.y}, a[2] = Pair{h.z, l.z}, a[3] = Pair{h.w, l.w};
    }
    for (int t = 0; t < b.slots - 1; ++t) {
      const float4 x = reinterpret_cast<const float4*>(b.ring + b.stride * ((b.folded + t) % b.slots))[q];
      a[0].add(x.x), a[1].add(x.y), a[2].add(x.z), a[3].add(x.w);
    }
    hi[q] = make_float4(a[0].hi, a[1].hi, a[2].hi, a[3].hi);
    lo[q] = make_float4(a[0].lo, a[1].lo, a[2].lo, a[3].lo);
  }
}

// The halves meet: score_j = sum_v [K + V t_H + (P - V) h_H], K = h_1 + .. + h_H, V = h_1 + .. +
// h_{L-H}. A thread takes four columns of a row (always the same four). Nothing beyond the stored vectors
// is rounded to FP32: sums over t, products and the thread's sum are kept as pairs, and summed in FP64
// over threads and blocks in a fixed order.
template <int C, bool WEIGHTED>
__global__ void __launch_bounds__(kThreads) batch_meet(const BatchVecs b, int32_t odd, int32_t n_active,
                                                       const BatchRow* __restrict__ row,
                                                       const BatchScale* __restrict__ scale, double* __restrict__ part,
                                                       unsigned* __restrict__ done, int32_t groups,
                                                       double* __restrict__ out) {
  constexpr int Q = C / 4;  // float4s of a row
  __shared__ double sm[kThreads][4];
  __shared__ int is_last;
  Pair acc[4] = {};
  const int64_t quads = static_cast<int64_t>(n_active) * Q;
  for (int64_t q = blockIdx.x * static_cast<int64_t>(kThreads) + threadIdx.x; q < quads;
       q += static_cast<int64_t>(gridDim.x) * kThreads) {
    const int32_t v = static_cast<int32_t>(q / Q);
    Pair k[4] = {};
    float h[4];
    if (b.folded > 0) {
      const float4 x = __ldcs(reinterpret_cast<const float4*>(b.V) + q);
      const float4 y = __ldcs(reinterpret_cast<const float4*>(b.V + b.stride) + q);
      k[0] = Pair{x.x, y.x}, k[1] = Pair{x.y, y.y}, k[2] = Pair{x.z, y.z}, k[3] = Pair{x.w, y.w};
    }
    for (int t = b.folded + 1; t < b.H; ++t) {
      const float4 x = __ldcs(reinterpret_cast<const float4*>(b.ring + b.stride * ((t - 1) % b.slots)) + q);
      k[0].add(x.x), k[1].add(x.y), k[2].add(x.z), k[3].add(x.w);
    }
    {
      const float4 x = __ldcs(reinterpret_cast<const float4*>(b.ring + b.stride * ((b.H - 1) % b.slots)) + q);
      h[0] = x.x, h[1] = x.y, h[2] = x.z, h[3] = x.w;
    }
    const float4 rw = __ldg(reinterpret_cast<const float4*>(row) + v);
    const Pair t{rw.x, rw.y}, p{rw.z, rw.w};
    Pair i{1.0f, 0.0f}, i2{1.0f, 0.0f};
    if constexpr (WEIGHTED) {
      const float4 sc = __ldg(reinterpret_cast<const float4*>(scale) + v);
      i = Pair{sc.x, sc.y}, i2 = Pair{sc.z, sc.w};
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      Pair kk = k[c];
      kk.add(h[c]);
      const Pair vv = odd ? k[c] : kk;
      Pair rest = p;
      rest.sub(vv);
      if constexpr (WEIGHTED) {
        acc[c].add(kk.times(i));
        acc[c].add(rest.pos().times(i2.times(h[c])));
      } else {
        acc[c].add(kk);
        acc[c].add(rest.pos().times(h[c]));
      }
      acc[c].add(vv.times(t));
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) sm[threadIdx.x][c] = acc[c].get();
  __syncthreads();
  if (threadIdx.x < C) {  // column threadIdx.x: the threads that hold its four
    double x = 0.0;
    for (int i = threadIdx.x / 4; i < kThreads; i += Q) x += sm[i][threadIdx.x & 3];
    part[static_cast<size_t>(blockIdx.x) * C + threadIdx.x] = x;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicInc(done, gridDim.x - 1) == gridDim.x - 1;  // back to 0 for the next
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  if (static_cast<int>(threadIdx.x) < groups) {
    double x = 0.0;
#pragma unroll 8
    for (int i = 0; i < static_cast<int>(gridDim.x); ++i) x += __ldcg(part + static_cast<size_t>(i) * C + threadIdx.x);
    out[threadIdx.x] = x;
  }
}
constexpr int kBatchMeetBlocks = 456;  // three per SM

int blocks_for(int64_t n, int per = 256) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((n + per - 1) / per, 152 * 32)));
}

}  // namespace

namespace {
// Waits for a stream when a call leaves early with an error, so that nothing it launched still
// runs when its buffers are reused or freed.
struct StreamGuard {
  cudaStream_t s;
  bool ok = false;
  ~StreamGuard() {
    if (!ok) {
      cudaStreamSynchronize(s);
      cudaGetLastError();
    }
  }
};
}  // namespace

gedwalk_status score_one(Graph& g, Workspace& ws, const std::vector<int32_t>& S_int, const Resolved& r,
                         double* score) {
  cudaStream_t s = r.stream;
  if (S_int.empty()) {
    *score = 0.0;
    return GEDWALK_OK;
  }
  if (!g.directed) {
    const gedwalk_status st = score_run(g, ws, S_int, r, score);
    if (st != GEDWALK_ERR_OOM) return st;
    // no memory for the half-length run's five vectors: sweeps of the full length keep two
  }
  StreamGuard guard{s};
  const size_t es = r.fp64 ? 8 : 4;
  const size_t vbytes = static_cast<size_t>(g.n) * 2 * es;
  GW_TRY(ws.x0.ensure(vbytes, s));
  GW_TRY(ws.x1.ensure(vbytes, s));
  GW_TRY(ensure_sweep_scratch(g, ws, 2, r.fp64, s));
  GW_TRY(ws.small.ensure(64, s));
  GW_TRY(upload_mask(g, ws, S_int, s));
  if (r.fp64)
    init_two_state<double><<<blocks_for(g.n), 256, 0, s>>>(ws.x0.as<double>(), ws.mask.as<uint32_t>(), g.n,
                                                           g.weighted ? g.rs_d.as<double>() : nullptr);
  else
    init_two_state<float><<<blocks_for(g.n), 256, 0, s>>>(ws.x0.as<float>(), ws.mask.as<uint32_t>(), g.n,
                                                          g.weighted ? g.rs_f.as<float>() : nullptr);
  GW_KCHECK();
  SweepArgs a = base_args(g, ws);
  a.alpha = r.alpha;
  void* cur = ws.x0.p;
  void* nxt = ws.x1.p;
  for (int32_t i = 1; i <= r.L; ++i) {
    a.X = cur;
    a.Y = nxt;
    a.accumulate = i > 1;
    GW_TRY(launch_sweep(MODE_SCORE, r.fp64, 2, a, s));
    std::swap(cur, nxt);
  }
  GW_TRY(reduce_slots(g, ws, 1, ws.small.as<double>(), s));
  double h = 0;
  GW_CUDA(cudaMemcpyAsync(&h, ws.small.p, sizeof h, cudaMemcpyDeviceToHost, s));
  GW_CUDA(cudaStreamSynchronize(s));
  *score = h;
  guard.ok = true;
  return GEDWALK_OK;
}

// Picks the column-block width with the lowest sweep time per column (timed on this graph). A
// gather fetches whole 32-byte sectors, so widths below 8 FP32 columns waste part of each; above
// 32 a sweep's pair of vectors of a 10^6-vertex graph outgrows the L2 and the per-column time rises (the
// tuning log records it). Only the dense sweep is timed: the meeting pass and a block's launches, a quarter
// of its time, favour wider blocks (Barabasi-Albert 10^6, 512 groups: 20.7 ms at the 16 columns it picks, 19.8
// at 32, 21.6 at 64).
gedwalk_status autotune_batch(Graph& g, Workspace& ws, const Resolved& r) {
  if (g.batch_cols > 0) return GEDWALK_OK;
  cudaStream_t s = r.stream;
  static const int kCand[] = {8, 16, 32, 64};
  double best = INFINITY;
  int best_c = 16;
  cudaEvent_t e0, e1;
  GW_CUDA(cudaEventCreate(&e0));
  GW_CUDA(cudaEventCreate(&e1));
  g.tune_log.clear();
  for (int c : kCand) {
    const size_t vec = static_cast<size_t>(g.n) * c;
    if (ws.xs.ensure(2 * vec * sizeof(float), s) != GEDWALK_OK) break;
    GW_TRY(ensure_sweep_scratch(g, ws, c, false, s));
    init_batch<<<blocks_for(static_cast<int64_t>(g.n) * c), 256, 0, s>>>(ws.xs.as<float>(), g.n, g.n, c, c);
    GW_KCHECK();
    SweepArgs a = base_args(g, ws);
    a.alpha = r.alpha;
    a.X = ws.xs.p;
    a.Y = ws.xs.as<float>() + vec;
    for (int w = 0; w < 2; ++w) GW_TRY(launch_sweep(MODE_PLAIN, false, c, a, s));
    const int reps = 5;
    GW_CUDA(cudaEventRecord(e0, s));
    for (int w = 0; w < reps; ++w) GW_TRY(launch_sweep(MODE_PLAIN, false, c, a, s));
    GW_CUDA(cudaEventRecord(e1, s));
    GW_CUDA(cudaEventSynchronize(e1));
    float ms = 0;
    GW_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    const double per_col = ms / reps / c;
    g.tune_log.emplace_back(c, per_col);
    if (per_col < best) {
      best = per_col;
      best_c = c;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  g.batch_cols = best_c;
  return GEDWALK_OK;
}

// Vectors of a batch's ring, and those it stores in all: x_1 .. x_H in the ring (x_0 of a weighted graph in
// its last slot); beyond the ring the oldest are folded into two vectors (hi, lo) behind it.
static int batch_ring(const Graph& g, int64_t C) {
  return static_cast<int64_t>(g.n_active) * C * 4 * kBatchRing > kWideBytes ? 2 : kBatchRing;
}
static int batch_stored(const Graph& g, int32_t L, int ring) {
  const int H = (L + 1) / 2;
  return H > ring ? ring + 2 : g.weighted ? ring : H;
}

int64_t score_batch_footprint(const Graph& g, int64_t members, int32_t groups, int32_t L) {
  const int64_t C = g.batch_cols > 0 ? g.batch_cols : 32;  // before tuning: the widest width tried
  const int64_t n = g.n;
  int64_t b = members * (4 + 4 + 8) + static_cast<int64_t>(groups + 1) * 4 + 256;  // members, columns, sums
  // the scratch fits the larger of a directed graph's two plans
  auto larger = [&](int32_t a, int32_t rev) { return static_cast<int64_t>(std::max({a, g.directed ? rev : 0, 1})); };
  b += larger(g.plan.num_slices, g.plan_r.num_slices) * C * 4 + larger(g.plan.num_heavy, g.plan_r.num_heavy) * 4;
  b += static_cast<int64_t>(groups) * 8 + 64 + (n + 31) / 32 * 4;
  if (!g.directed) {
    b += static_cast<int64_t>(g.n_active) * C * 4 * batch_stored(g, L, batch_ring(g, C));
    b += n * (g.weighted ? 32 : 16) + (kBatchMeetBlocks * C + 1) * 8;
    return b;
  }
  b += 2 * n * C * 4;  // walk vectors x0, x1
  b += larger(g.plan.num_slots, g.plan_r.num_slots) * C * 8 + C * kReduceParts * 8;
  return b;
}

// The blocks of an undirected graph's batch; the members (rows, columns) are on the device, the scores
// go to ws.small. The table holds rows 0..H (the caller keeps its lock).
static gedwalk_status batch_runs(Graph& g, Workspace& ws, int C, int ring_slots, const int32_t* offsets, int32_t G, const int32_t* mrow,
                                 const int32_t* mcol, const Resolved& r, cudaStream_t s) {
  if (g.n_active == 0) {  // no edges, no walks
    GW_CUDA(cudaMemsetAsync(ws.small.p, 0, sizeof(double) * G, s));
    return GEDWALK_OK;
  }
  const int32_t L = r.L, H = (L + 1) / 2;
  const int64_t vec = static_cast<int64_t>(g.n_active) * C;
  GW_TRY(ws.tail.ensure(static_cast<size_t>(g.n) * sizeof(BatchRow), s));
  if (g.weighted) GW_TRY(ws.bound.ensure(static_cast<size_t>(g.n) * sizeof(BatchScale), s));
  const size_t nz_bytes = (static_cast<size_t>(g.n) + 31) / 32 * sizeof(uint32_t);
  GW_TRY(ws.mask.ensure(nz_bytes, s));
  uint32_t* nz = ws.mask.as<uint32_t>();
  GW_TRY(ws.partial.ensure(static_cast<size_t>(std::max(g.plan.num_slices, 1)) * C * sizeof(float), s));
  const size_t cbytes = static_cast<size_t>(std::max(g.plan.num_heavy, 1)) * sizeof(unsigned);
  if (ws.counters.bytes < cbytes || !ws.counters.p) GW_TRY(ws.counters.ensure(cbytes, s, /*zero=*/true));
  GW_TRY(ws.parts.ensure((static_cast<size_t>(kBatchMeetBlocks) * C + 1) * sizeof(double), s));
  double* part = ws.parts.as<double>() + 1;
  unsigned* done = ws.parts.as<unsigned>();
  GW_CUDA(cudaMemsetAsync(done, 0, sizeof(double), s));
  const double* T = g.ttab.as<double>();
  BatchRow* row = ws.tail.as<BatchRow>();
  BatchScale* scale = ws.bound.as<BatchScale>();
  batch_totals<<<blocks_for(g.n_active), 256, 0, s>>>(T, g.n, g.n_active, L, H, g.weighted ? g.rs_d.as<double>() : nullptr,
                                                      row, scale);
  GW_KCHECK();
  float* ring = ws.xs.as<float>();
  auto slot = [&](int32_t t) { return ring + vec * ((t + ring_slots - 1) % ring_slots); };  // x_0: the last slot
  float* V = ring + vec * ring_slots;
  SweepArgs a = base_args(g, ws);
  a.alpha = r.alpha;
  const int meet = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(kBatchMeetBlocks, (vec / 4 + kThreads - 1) / kThreads)));
  for (int32_t g0 = 0; g0 < G; g0 += C) {
    const int32_t g1 = std::min(G, g0 + C);
    const int32_t m0 = offsets[g0], cnt = offsets[g1] - m0;
    auto own = [&](int32_t t, uint32_t* bits) -> gedwalk_status {
      if (cnt == 0) return GEDWALK_OK;
      batch_own<<<blocks_for(cnt), 256, 0, s>>>(slot(t), C, mrow + m0, mcol + m0, cnt, T + static_cast<size_t>(t) * g.n,
                                                g.n_active, bits);
      GW_KCHECK();
      return GEDWALK_OK;
    };
    int32_t t = g.weighted ? 0 : 1;  // the first vector: x_0 = the groups' indicators, or x_1 from counts
    GW_CUDA(cudaMemsetAsync(slot(t), 0, static_cast<size_t>(vec) * sizeof(float), s));
    GW_CUDA(cudaMemsetAsync(nz, 0, nz_bytes, s));
    if (!g.weighted && cnt > 0) {
      batch_scatter<<<dim3(static_cast<unsigned>(std::min((cnt + 7) / 8, 2048)), g.dmax > kScatterRow ? 32 : 1), 256, 0, s>>>(
          reinterpret_cast<int32_t*>(slot(1)), C, mrow + m0, mcol + m0, cnt, a.rp, a.ci, nz);
      GW_KCHECK();
      batch_count_scale<<<blocks_for(g.n_active), 256, 0, s>>>(slot(1), C, g.n_active, static_cast<float>(r.alpha), nz);
      GW_KCHECK();
    }
    GW_TRY(own(t, nz));
    a.nz = nz;  // the first vector is zero but next to the groups: its sweep gathers those rows alone
    BatchVecs b{ring, vec, ring_slots, V, 0, H};
    for (++t; t <= H; ++t) {
      if (t - b.folded > ring_slots) {  // x_t takes the slot of x_{t-slots}: fold all before x_{t-1}
        batch_fold<<<blocks_for(vec / 4), 256, 0, s>>>(b, vec / 4);
        GW_KCHECK();
        b.folded += ring_slots - 1;
      }
      a.X = slot(t - 1);
      a.Y = slot(t);
      GW_TRY(launch_sweep(MODE_PLAIN, false, C, a, s));
      a.nz = nullptr;
      GW_TRY(own(t, nullptr));
    }
    double* out = ws.small.as<double>() + g0;
#define GW_MEET(CC)                                                                                                     \
  if (C == CC) {                                                                                                        \
    if (g.weighted)                                                                                                     \
      batch_meet<CC, true><<<meet, kThreads, 0, s>>>(b, L & 1, g.n_active, row, scale, part, done, g1 - g0, out);       \
    else                                                                                                                \
      batch_meet<CC, false><<<meet, kThreads, 0, s>>>(b, L & 1, g.n_active, row, nullptr, part, done, g1 - g0, out);    \
  }
    GW_MEET(4) GW_MEET(8) GW_MEET(16) GW_MEET(32) GW_MEET(64)
#undef GW_MEET
    GW_KCHECK();
  }
  return GEDWALK_OK;
}

gedwalk_status score_batch_impl(Graph& g, Workspace& ws, const int32_t* offsets, const int32_t* members_int,
                                int32_t G, const Resolved& r, double* scores) {
  cudaStream_t s = r.stream;
  if (G == 0) return GEDWALK_OK;
  StreamGuard guard{s};
  // the caller has made the walk-total table for alpha and L, and tuned the width
  std::shared_lock<std::shared_mutex> rl(g.tt_lock);
  if (g.tt_alpha != r.alpha || g.tt_rows < walk_rows(g, r.L + 1) || g.batch_cols <= 0)
    return fail(GEDWALK_ERR_INVALID, "walk-total table or column width not prepared for this batch");
  int C = g.batch_cols;
  int ring = 0;
  if (!g.directed) {
    // the stored vectors, with a shorter ring and then narrower blocks where the device cannot hold them
    // (at four columns as much as two vectors of eight, the least that full-length sweeps would take)
    for (ring = batch_ring(g, C);;) {
      const size_t vec = static_cast<size_t>(g.n_active) * C * sizeof(float);
      const gedwalk_status st = ws.xs.ensure(vec * batch_stored(g, r.L, ring), s);
      if (st == GEDWALK_OK) break;
      if (st != GEDWALK_ERR_OOM || (ring == 2 && C == 4)) return st;
      if (ring > 2) ring = 2;
      else C /= 2;
    }
  }
  const int64_t total = offsets[G];
  // members: row (internal id), column within its block, accumulator; group offsets
  const size_t mbytes = static_cast<size_t>(total) * (4 + 4 + 8) + static_cast<size_t>(G + 1) * 4 + 256;
  GW_TRY(ws.members.ensure(mbytes, s));
  char* base = ws.members.as<char>();
  double* acc = reinterpret_cast<double*>(base);
  int32_t* mrow = reinterpret_cast<int32_t*>(acc + total);
  int32_t* mcol = mrow + total;
  int32_t* goff = mcol + total;
  // members, their columns and the group offsets go up in one copy from pinned staging
  const size_t up = sizeof(int32_t) * (2 * static_cast<size_t>(total) + G + 1);
  GW_TRY(ws.ensure_pinned(std::max(up, sizeof(double) * static_cast<size_t>(G)) + 64));
  int32_t* hst = static_cast<int32_t*>(ws.pinned);
  if (total > 0) memcpy(hst, members_int, sizeof(int32_t) * total);
  for (int32_t j = 0; j < G; ++j)
    for (int32_t i = offsets[j]; i < offsets[j + 1]; ++i) hst[total + i] = j % C;
  memcpy(hst + 2 * total, offsets, sizeof(int32_t) * (G + 1));
  GW_CUDA(cudaMemcpyAsync(mrow, hst, up, cudaMemcpyHostToDevice, s));
  GW_TRY(ws.small.ensure(static_cast<size_t>(G) * sizeof(double) + 64, s));
  const double* T = g.ttab.as<double>();
  if (!g.directed) {
    GW_TRY(batch_runs(g, ws, C, ring, offsets, G, mrow, mcol, r, s));
    GW_CUDA(cudaMemcpyAsync(ws.pinned, ws.small.p, sizeof(double) * G, cudaMemcpyDeviceToHost, s));
    GW_CUDA(cudaStreamSynchronize(s));
    memcpy(scores, ws.pinned, sizeof(double) * G);
    guard.ok = true;
    return GEDWALK_OK;
  }
  const size_t vbytes = static_cast<size_t>(g.n) * C * 4;
  GW_TRY(ws.x0.ensure(vbytes, s));
  GW_TRY(ws.x1.ensure(vbytes, s));
  GW_TRY(ensure_sweep_scratch(g, ws, C, false, s));
  SweepArgs a = base_args(g, ws);
  a.alpha = r.alpha;
  if (g.n_active < g.n)
    GW_CUDA(cudaMemsetAsync(ws.x1.as<float>() + static_cast<size_t>(g.n_active) * C, 0,
                            sizeof(float) * C * (static_cast<size_t>(g.n) - g.n_active), s));
  if (total > 0) {
    batch_member_init<<<blocks_for(total), 256, 0, s>>>(mrow, acc, static_cast<int32_t>(total), T, g.n, r.L);
    GW_KCHECK();
  }
  for (int32_t g0 = 0; g0 < G; g0 += C) {
    const int32_t g1 = std::min(G, g0 + C);
    const int32_t m0 = offsets[g0], m1 = offsets[g1];
    const int32_t cnt = m1 - m0;
    init_batch<<<blocks_for(static_cast<int64_t>(g.n) * C), 256, 0, s>>>(ws.x0.as<float>(), g.n, g.n_active, C,
                                                                          g1 - g0);
    GW_KCHECK();
    if (cnt > 0) {
      zero_members<<<blocks_for(cnt), 256, 0, s>>>(ws.x0.as<float>(), C, mrow + m0, mcol + m0, cnt);
      GW_KCHECK();
    }
    void* cur = ws.x0.p;
    void* nxt = ws.x1.p;
    for (int32_t p = 1; p <= r.L; ++p) {
      a.X = cur;
      a.Y = nxt;
      GW_TRY(launch_sweep(MODE_PLAIN, false, C, a, s));
      if (cnt > 0) {
        batch_member_epilogue<<<blocks_for(cnt), 256, 0, s>>>(static_cast<float*>(nxt), C, mrow + m0, mcol + m0,
                                                               acc + m0, cnt, T, g.n, r.L - p);
        GW_KCHECK();
      }
      std::swap(cur, nxt);
    }
  }
  batch_group_sum<<<blocks_for(G), 256, 0, s>>>(acc, goff, G, ws.small.as<double>());
  GW_KCHECK();
  GW_CUDA(cudaMemcpyAsync(ws.pinned, ws.small.p, sizeof(double) * G, cudaMemcpyDeviceToHost, s));
  GW_CUDA(cudaStreamSynchronize(s));
  memcpy(scores, ws.pinned, sizeof(double) * G);
  guard.ok = true;
  return GEDWALK_OK;
}

}  // namespace gw

using namespace gw;

extern "C" {

gedwalk_status gedwalk_score(gedwalk_graph_t h, const int32_t* S, int32_t s_len, const gedwalk_params* params,
                             double* score, int32_t* L_used, double* tail_bound) {
  if (!h || !score) return fail(GEDWALK_ERR_INVALID, "graph or score is NULL");
  Graph* g = G(h);
  std::lock_guard<std::mutex> lk(g->mu);
  GW_CUDA(cudaSetDevice(g->device));
  std::vector<int32_t> S_int;
  GW_TRY(map_group(*g, S, s_len, &S_int));
  Resolved r;
  GW_TRY(resolve(*g, params, 0.0, &r));
  double v = 0;
  GW_TRY(score_one(*g, g->ws, S_int, r, &v));
  *score = v;
  if (L_used) *L_used = r.L;
  if (tail_bound) *tail_bound = r.bound;
  return GEDWALK_OK;
}

gedwalk_status gedwalk_batch_tuning(gedwalk_graph_t h, int32_t* cols, double* us_per_col, int32_t cap, int32_t* count,
                                    int32_t* chosen) {
  if (!h) return fail(GEDWALK_ERR_INVALID, "graph is NULL");
  if (cap < 0 || (cap > 0 && (!cols || !us_per_col))) return fail(GEDWALK_ERR_INVALID, "NULL output or cap < 0");
  Graph* g = gw::G(h);
  std::lock_guard<std::mutex> lk(g->mu);
  const int32_t m = static_cast<int32_t>(g->tune_log.size());
  for (int32_t j = 0; j < std::min(m, cap); ++j) {
    cols[j] = g->tune_log[j].first;
    us_per_col[j] = g->tune_log[j].second * 1e3;
  }
  if (count) *count = m;
  if (chosen) *chosen = g->batch_cols;
  return GEDWALK_OK;
}

gedwalk_status gedwalk_batch_set_width(gedwalk_graph_t h, int32_t cols) {
  if (!h) return fail(GEDWALK_ERR_INVALID, "graph is NULL");
  if (!(cols == 0 || cols == 8 || cols == 16 || cols == 32 || cols == 64))
    return fail(GEDWALK_ERR_INVALID, "column-block width must be 0 (tune), 8, 16, 32 or 64");
  Graph* g = gw::G(h);
  std::lock_guard<std::mutex> lk(g->mu);
  g->batch_cols = cols;
  return GEDWALK_OK;
}

gedwalk_status gedwalk_score_batch(gedwalk_graph_t h, const int32_t* offsets, const int32_t* members, int32_t G,
                                   const gedwalk_params* params, double* scores, int32_t* L_used) {
  if (!h || (G > 0 && (!offsets || !scores))) return fail(GEDWALK_ERR_INVALID, "NULL argument");
  if (G < 0) return fail(GEDWALK_ERR_INVALID, "G must be >= 0");
  Graph* g = gw::G(h);
  std::lock_guard<std::mutex> lk(g->mu);
  GW_CUDA(cudaSetDevice(g->device));
  if (G > 0 && offsets[0] != 0) return fail(GEDWALK_ERR_INVALID, "offsets[0] must be 0");
  // map and deduplicate each group (set semantics), rebuilding the offsets
  std::vector<int32_t> off(static_cast<size_t>(G) + 1, 0), mem, tmp;
  for (int32_t j = 0; j < G; ++j) {
    if (offsets[j + 1] < offsets[j]) return fail(GEDWALK_ERR_INVALID, "offsets decrease at group %d", j);
    GW_TRY(map_group(*g, members + offsets[j], offsets[j + 1] - offsets[j], &tmp));
    mem.insert(mem.end(), tmp.begin(), tmp.end());
    off[j + 1] = static_cast<int32_t>(mem.size());
  }
  Resolved r;
  GW_TRY(resolve(*g, params, 0.0, &r));
  r.fp64 = false;
  GW_TRY(ensure_totals(*g, r.alpha, r.L + 1, r.stream));
  GW_TRY(autotune_batch(*g, g->ws, r));
  GW_TRY(score_batch_impl(*g, g->ws, off.data(), mem.data(), G, r, scores));
  if (L_used) *L_used = r.L;
  return GEDWALK_OK;
}

}  // extern "C"
