// Greedy GED-Walk maximisation (problem (ii), Def. ged-max; Prop. greedy_approx) and
// all-vertex exact marginal gains.
//
// Undirected graphs: runs of half the walk length (run.cu). A chain run carries the next steps'
// guessed winners c_1..c_D, each under S and the earlier ones, and brings for every level the best
// upper bounds of the unevaluated vertices and the exact gain of its guess. A step takes the guess
// once no bound (inflated by the rounding tolerance) reaches its gain; otherwise the best-bounded
// vertices are evaluated exactly, side by side under S, until the best exact gain is beyond every
// bound. No result depends on the guesses. A vertex whose bound is exactly 0 has gain exactly 0.
// Among equal gains the lowest caller id wins.
//
// Directed graphs (maximize_directed): a step with current group S runs L fused sweeps (phi^miss_1..L
// under S in column 0, stored in a table, and the exact gains of speculative candidates), the psi^miss
// sweeps of the other orientation on the reverse CSR, and one pass over all vertices with the
// Lemma-initialize bound
//       ub(x) = sum_{i=1..L} alpha^i P_i(S, x) = sum_{1 <= a+b <= L} y_a(x) z_b(x),
// y_a = alpha^a phi^miss_a, z_b = alpha^b psi^miss_b, min'd with the last exact gain; then the same
// certification.
// The gain of candidate c counts walks of length 1..L in G[V\S] through c
// (proof of Prop. ged_submod): h_0 = e_c, h_t = alpha 1_{V\S} . A h_{t-1} except
// h_t(c) = phi^miss_t(c); gain = sum_t sum_v h_t(v) in FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>

#include "run.h"

namespace gw {
namespace {

constexpr int kSelPerSM = 4;               // resident blocks of the bound pass per SM
constexpr int kSelU = 2;                   // vertices per lane and iteration of the bound pass
constexpr int kSelBlocks = 152 * kSelPerSM;

struct SelOut {  // device -> host after each selection pass
  float val[kTopK];
  int32_t id[kTopK];
  // the unevaluated vertex with bound exactly 0 and the smallest caller id, packed as
  // (caller id << 32) | internal id (all ones: none)
  unsigned long long zero_min;
  int32_t sampled;  // stochastic greedy: sampled vertices outside S seen by the pass
  int32_t done;     // blocks of the pass that have finished
  double gains[16];  // exact gains of the last candidate batch
};

// Sampling of one selection pass; thr == UINT64_MAX means every vertex takes part.
struct Sampling {
  uint64_t thr;
  uint64_t seed;
  uint32_t step;
};

// mtab row 0 = phi^miss_0 = 1_{V\S}; X column 0 (fused) = the same; candidate columns = e_c.
template <typename T>
__global__ void greedy_init(T* __restrict__ m0, T* __restrict__ X, int cols, int first_cand_col,
                            const int32_t* __restrict__ cand, const uint32_t* __restrict__ mask, int32_t n) {
  __shared__ int sc[16];
  if (threadIdx.x < 16) sc[threadIdx.x] = threadIdx.x < cols - first_cand_col ? cand[threadIdx.x] : -1;
  __syncthreads();
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const bool inS = (mask[v >> 5] >> (v & 31)) & 1u;
    const T m = inS ? T(0) : T(1);
    if (m0) m0[v] = m;
    T* row = X + static_cast<size_t>(v) * cols;
    if (first_cand_col == 1) row[0] = m;
    for (int j = first_cand_col; j < cols; ++j) row[j] = (sc[j - first_cand_col] == v) ? T(1) : T(0);
  }
}

__global__ void update_stale(Stale* __restrict__ stale, const int32_t* __restrict__ cand,
                             const double* __restrict__ gains, int count, int32_t step, double* __restrict__ out) {
  const int j = threadIdx.x;
  if (j >= count) return;
  const int c = cand[j];
  if (out) out[j] = gains[j];
  if (c < 0) return;
  Stale st;
  st.ub = __double2float_ru(gains[j]);
  st.step = step;
  stale[c] = st;
}

__device__ __forceinline__ float to_f32_up(float v) { return v; }
__device__ __forceinline__ float to_f32_up(double v) { return __double2float_ru(v); }

// Lemma-initialize bound of vertex x:
//   ub(x) = sum_{i=1..L} alpha^i P_i(S, x) = sum over ordered pairs 1 <= a+b <= L of y_a(x) z_b(x)
//         = y_0 (Q_L - z_0) + sum_{a=1..L} y_a Q_{L-a},   Q_q = sum_{b <= q} z_b,
// y_a = alpha^a phi^miss_a(x) and z_b = alpha^b psi^miss_b(x), the S-avoiding walks in the other
// orientation (a directed graph's reverse; on an undirected graph z = y, zcol == col). Evaluated
// in FP32 with every operation rounded toward +infinity on non-negative inputs (FP64 inputs are
// first rounded up), so the result never falls below the bound of the stored vectors.
template <typename T, int L>
__device__ __forceinline__ float ub_fixed(const T* __restrict__ col, const T* __restrict__ zcol, int32_t n, float m0) {
  // row 0 is phi^miss_0 = psi^miss_0 = 1_{V\S}: m0, not read from the tables
  float y[L + 1], z[L + 1];
  y[0] = m0;
#pragma unroll
  for (int a = 1; a <= L; ++a) y[a] = to_f32_up(__ldcs(col + static_cast<size_t>(a) * n));
  if (zcol == col) {
#pragma unroll
    for (int a = 0; a <= L; ++a) z[a] = y[a];
  } else {
    z[0] = m0;
#pragma unroll
    for (int a = 1; a <= L; ++a) z[a] = to_f32_up(__ldcs(zcol + static_cast<size_t>(a) * n));
  }
  float Q[L + 1];
  Q[0] = z[0];
  float R = 0.0f;
#pragma unroll
  for (int q = 1; q <= L; ++q) {
    Q[q] = __fadd_ru(Q[q - 1], z[q]);
    R = __fadd_ru(R, z[q]);
  }
  float ub = __fmul_ru(y[0], R);
#pragma unroll
  for (int a = 1; a <= L; ++a) ub = __fmaf_ru(y[a], Q[L - a], ub);
  return ub;
}

// The same sum for any L in one pass: a runs down from L while Q_{L-a} = z_0 + ... + z_{L-a}
// grows, so every pair (a, b) with 1 <= a + b <= L is met once: y_a Q_{L-a} for a >= 1, and
// y_0 (Q_L - z_0) at the end. Two table reads per step, every operation rounded up.
template <typename T>
__device__ float ub_any(const T* __restrict__ col, const T* __restrict__ zcol, int32_t n, int32_t L, float m0) {
  float Q = m0;     // Q_0 = z_0
  float R = 0.0f;   // z_1 + ... + z_{L-a}
  float ub = 0.0f;
  for (int a = L; a >= 1; --a) {
    if (a < L) {
      const float zb = to_f32_up(__ldcs(zcol + static_cast<size_t>(L - a) * n));
      Q = __fadd_ru(Q, zb);
      R = __fadd_ru(R, zb);
    }
    ub = __fmaf_ru(to_f32_up(__ldcs(col + static_cast<size_t>(a) * n)), Q, ub);
  }
  R = __fadd_ru(R, to_f32_up(__ldcs(zcol + static_cast<size_t>(L) * n)));
  return __fmaf_ru(m0, R, ub);
}

// Lemma-initialize bound + selection over vertices [0, n_scan) (the tables have n rows apart):
// the kTopK unevaluated vertices outside S with the largest bounds go to out->val / out->id.
// Each warp keeps its own list (bounds offered 32 at a time, two per lane per iteration), a block
// merges its warps' lists into sel_v / sel_id[block], and the last block to finish merges the
// blocks' lists: only the kTopK blocks whose heads rank among the best kTopK heads can hold an
// entry of the result (any other head has kTopK better entries ahead of it). out->done counts the
// finished blocks (0 before the pass). LF = L when L <= 16, else 0 (any L).
template <typename T, int LF>
__global__ void __launch_bounds__(kThreads, kSelPerSM) ub_select(const T* __restrict__ mtab, const T* __restrict__ ztab,
                                                     int32_t L, int32_t n, int32_t n_scan,
                                                     const uint32_t* __restrict__ mask,
                                                     const Stale* __restrict__ stale, int32_t step,
                                                     const int32_t* __restrict__ perm, float* __restrict__ sel_v,
                                                     int* __restrict__ sel_id, SelOut* __restrict__ out,
                                                     const Sampling smp) {
  constexpr int NW = kThreads / 32;
  static_assert(2 * NW >= kTopK, "the final merge gives each warp two block lists");
  constexpr int U = kSelU;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int nsampled = 0;
  WarpList w;
  // U * 32 consecutive vertices per warp and iteration, all loads issued before any decision
  const int32_t wid = blockIdx.x * NW + warp;
  const int32_t wstride = gridDim.x * NW * (U * 32);
  for (int32_t base = wid * (U * 32); base < n_scan; base += wstride) {
    float b[U];
    bool live[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int32_t xr = base + k * 32 + lane;
      const int32_t x = xr < n_scan ? xr : n_scan - 1;
      const bool inS = (__ldg(mask + (x >> 5)) >> (x & 31)) & 1u;
      const Stale st = stale[x];
      const float m0 = inS ? 0.0f : 1.0f;
      float ub = LF > 0 ? ub_fixed<T, (LF > 0 ? LF : 1)>(mtab + x, ztab + x, n, m0)
                        : ub_any<T>(mtab + x, ztab + x, n, L, m0);
      if (st.step >= 0 && st.ub < ub) ub = st.ub;
      b[k] = ub;
      bool in_sample = true;
      if (smp.thr != ~0ull && xr < n_scan && !inS)
        in_sample = sample_hash(smp.seed, smp.step, static_cast<uint32_t>(__ldg(perm + x))) < smp.thr;
      if (xr < n_scan && !inS && in_sample) ++nsampled;
      // evaluated with the current S: its exact gain is known
      live[k] = xr < n_scan && !inS && in_sample && st.step != step;
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int32_t x = base + k * 32 + lane;
      if (live[k] && b[k] == 0.0f)
        atomicMin(&out->zero_min, (static_cast<unsigned long long>(__ldg(perm + x)) << 32) | static_cast<uint32_t>(x));
      warp_list_offer(w, live[k] && b[k] != 0.0f, b[k], x, 0);
    }
  }
  if (smp.thr != ~0ull) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nsampled += __shfl_xor_sync(kFullMask, nsampled, o);
    if (lane == 0 && nsampled) atomicAdd(&out->sampled, nsampled);
  }
  __shared__ float sv[NW * kTopK];
  __shared__ int si[NW * kTopK], st[NW * kTopK];
  __shared__ int is_last;
  block_list_merge<NW>(w, sv, si, st);
  if (warp == 0) {
    if (lane < kTopK) {
      sel_v[blockIdx.x * kTopK + lane] = w.v;
      sel_id[blockIdx.x * kTopK + lane] = w.id;
    }
    __threadfence();
    __syncwarp();
    int done = 0;
    if (lane == 0) done = atomicAdd(&out->done, 1);
    if (lane == 0) is_last = done == static_cast<int>(gridDim.x) - 1;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  // the best kTopK block heads (tag: the block)
  WarpList h;
  for (int32_t b0 = warp * 32; b0 < static_cast<int32_t>(gridDim.x); b0 += NW * 32) {
    const int32_t blk = b0 + lane;
    const bool ok = blk < static_cast<int32_t>(gridDim.x);
    const float x = ok ? __ldcg(sel_v + static_cast<size_t>(blk) * kTopK) : -1.0f;
    const int ix = ok ? __ldcg(sel_id + static_cast<size_t>(blk) * kTopK) : INT_MAX;
    warp_list_offer(h, ix != INT_MAX, x, ix, blk);
  }
  block_list_merge<NW>(h, sv, si, st);
  __shared__ int heads[kTopK];
  if (warp == 0 && lane < kTopK) heads[lane] = h.id != INT_MAX ? h.tag : -1;
  __syncthreads();
  // the entries of those blocks, two block lists per warp
  WarpList f;
  {
    const int j = 2 * warp + (lane >> 4);
    const int blk = j < kTopK ? heads[j] : -1;
    const bool ok = blk >= 0;
    const size_t e = static_cast<size_t>(ok ? blk : 0) * kTopK + (lane & 15);
    const float x = ok ? __ldcg(sel_v + e) : -1.0f;
    const int ix = ok ? __ldcg(sel_id + e) : INT_MAX;
    warp_list_offer(f, ix != INT_MAX, x, ix, 0);
  }
  block_list_merge<NW>(f, sv, si, st);
  if (warp == 0 && lane < kTopK) {
    out->val[lane] = f.v;
    out->id[lane] = f.id;
  }
}

template <typename T>
cudaError_t launch_ub_select(int nb, cudaStream_t s, const T* mtab, const T* ztab, int32_t L, int32_t n,
                             int32_t n_scan, const uint32_t* mask,
                             const Stale* stale, int32_t step, const int32_t* perm, float* sel_v, int* sel_id,
                             SelOut* out, const Sampling& smp) {
#define GW_UB(LL)                                                                                          \
  case LL:                                                                                                 \
    ub_select<T, LL><<<nb, kThreads, 0, s>>>(mtab, ztab, L, n, n_scan, mask, stale, step, perm, sel_v, sel_id, \
                                             out, smp);                 \
    break;
  switch (L) {
    GW_UB(1) GW_UB(2) GW_UB(3) GW_UB(4) GW_UB(5) GW_UB(6) GW_UB(7) GW_UB(8)
    GW_UB(9) GW_UB(10) GW_UB(11) GW_UB(12) GW_UB(13) GW_UB(14) GW_UB(15) GW_UB(16)
    default:
      ub_select<T, 0><<<nb, kThreads, 0, s>>>(mtab, ztab, L, n, n_scan, mask, stale, step, perm, sel_v, sel_id,
                                              out, smp);
  }
#undef GW_UB
  return cudaGetLastError();
}

// Blocks of a selection pass: one wave at kSelPerSM blocks per SM, one iteration per lane at least.
int sel_blocks(int32_t n_scan) {
  constexpr int64_t per_block = int64_t(kThreads) * kSelU;
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(kSelBlocks, (int64_t(n_scan) + per_block - 1) / per_block)));
}

// Resets the per-pass counters of a selection pass.
__global__ void reset_selection(SelOut* out) {
  out->zero_min = kNoZero;
  out->sampled = 0;
  out->done = 0;
}

int blocks_for(int64_t n) { return static_cast<int>(std::min<int64_t>((n + 255) / 256, 152 * 16)); }

// Rows 1..L of the phi^miss table at isolated vertices: the sweeps never write them (no walk
// of length >= 1 ends there), so they are set to 0 once.
gedwalk_status zero_isolated_tail(Graph& g, void* tab, size_t es, int32_t L, cudaStream_t s) {
  if (g.n_active >= g.n || L < 1) return GEDWALK_OK;
  char* base = static_cast<char*>(tab) + static_cast<size_t>(g.n) * es + static_cast<size_t>(g.n_active) * es;
  GW_CUDA(cudaMemset2DAsync(base, static_cast<size_t>(g.n) * es, 0, static_cast<size_t>(g.n - g.n_active) * es, L, s));
  return GEDWALK_OK;
}

struct Cand {
  double g;
  int32_t v;       // internal id
  int32_t caller;  // caller id
};
// exact-gain order: larger gain first, then the lower caller id
bool cand_before(const Cand& a, const Cand& b) { return a.g > b.g || (a.g == b.g && a.caller < b.caller); }

struct GreedyCtx {
  Graph& g;
  Workspace& ws;
  const Resolved& r;
  cudaStream_t s;
  int32_t L;
  size_t es;
  SelOut* d_out;
  int32_t* d_cand;
  double* d_gains;
  SelOut* h_out;
  int64_t sweeps = 0;
};

// Issues init + L sweeps + column-sum reduction on c.s. ev (optional): two external events around
// the run of sweeps (graph capture; event nodes between kernel nodes cost a few microseconds each).
// rev (MODE_FUSED with one column): the sweeps run on the reverse CSR and fill the psi^miss table.
gedwalk_status issue_sweeps(GreedyCtx& c, int mode, int cols, bool profile, const std::vector<cudaEvent_t>* ev,
                            bool rev) {
  Graph& g = c.g;
  Workspace& ws = c.ws;
  const bool fp64 = c.r.fp64;
  const int first = mode == MODE_FUSED ? 1 : 0;
  DevBuf& tab = rev ? ws.ztab : ws.mtab;
  void* m0 = mode == MODE_FUSED ? tab.p : nullptr;
  if (fp64)
    greedy_init<double><<<blocks_for(g.n), 256, 0, c.s>>>(static_cast<double*>(m0), ws.x0.as<double>(), cols, first,
                                                           c.d_cand, ws.mask.as<uint32_t>(), g.n);
  else
    greedy_init<float><<<blocks_for(g.n), 256, 0, c.s>>>(static_cast<float*>(m0), ws.x0.as<float>(), cols, first,
                                                          c.d_cand, ws.mask.as<uint32_t>(), g.n);
  GW_KCHECK();
  SweepArgs a = rev ? base_args_rev(g, ws) : base_args(g, ws);
  a.alpha = c.r.alpha;
  a.cand = c.d_cand;
  void* cur = ws.x0.p;
  void* nxt = ws.x1.p;
  if (ev) GW_CUDA(cudaEventRecordWithFlags((*ev)[0], c.s, cudaEventRecordExternal));
  for (int32_t t = 1; t <= c.L; ++t) {
    a.X = cur;
    a.Y = nxt;
    a.accumulate = t > 1;
    char* row = tab.as<char>() + static_cast<size_t>(t) * g.n * c.es;
    if (mode == MODE_FUSED) a.Mout = row;
    else a.Min = row;
    GW_TRY(launch_sweep(mode, fp64, cols, a, c.s, profile));
    std::swap(cur, nxt);
  }
  if (ev) GW_CUDA(cudaEventRecordWithFlags((*ev)[1], c.s, cudaEventRecordExternal));
  const int nsum = sweep_sums(mode, cols);
  if (nsum > 0) GW_TRY(reduce_slots(g, ws, nsum, c.d_gains, c.s, rev));
  return GEDWALK_OK;
}

// Runs L sweeps. mode MODE_FUSED (column 0 = phi^miss, table rows written) or MODE_CAND.
gedwalk_status run_sweeps(GreedyCtx& c, int mode, int cols, const std::vector<int32_t>& cand, bool rev = false) {
  Graph& g = c.g;
  Workspace& ws = c.ws;
  const bool fp64 = c.r.fp64;
  int32_t hc[16];
  for (int j = 0; j < 16; ++j) hc[j] = j < static_cast<int>(cand.size()) ? cand[j] : -1;
  GW_CUDA(cudaMemcpyAsync(c.d_cand, hc, sizeof hc, cudaMemcpyHostToDevice, c.s));
  const size_t vbytes = static_cast<size_t>(g.n) * cols * c.es;
  GW_TRY(ws.x0.ensure(vbytes, c.s));
  GW_TRY(ws.x1.ensure(vbytes, c.s));
  GW_TRY(ensure_sweep_scratch(g, ws, cols, fp64, c.s));
  c.sweeps += c.L;
  if (g.plan.num_units == 0) return issue_sweeps(c, mode, cols, true, nullptr, rev);
  uint64_t abits;
  memcpy(&abits, &c.r.alpha, 8);
  auto bits = [](const void* p) { return static_cast<uint64_t>(reinterpret_cast<uintptr_t>(p)); };
  Sequence q;
  q.key = mix_all({uint64_t(mode), uint64_t(cols), uint64_t(fp64), uint64_t(c.L), uint64_t(g.n), uint64_t(rev), abits,
                   bits(ws.ztab.p), bits(&g), bits(c.s), bits(ws.x0.p), bits(ws.x1.p), bits(ws.mtab.p), bits(ws.slots.p),
                   bits(ws.parts.p), bits(ws.partial.p), bits(ws.counters.p), bits(ws.mask.p), bits(c.d_cand),
                   bits(c.d_gains)});
  q.kernels = 1 + c.L + (sweep_sums(mode, cols) > 0 ? 2 : 0);
  q.sweeps = c.L;
  q.bytes = sweep_bytes(mode, fp64, cols, g.n, g.nnz);
  q.prof_key = (mode * 1000 + cols) * 2 + (fp64 ? 1 : 0);
  return run_sequence(ws, c.s, q, [&](bool profile, const std::vector<cudaEvent_t>* ev) {
    return issue_sweeps(c, mode, cols, profile, ev, rev);
  });
}

}  // namespace

gedwalk_status greedy_shape(const Graph& g, const Resolved& r, int32_t flags, GreedyShape* out) {
  GreedyShape sh{};
  const bool adaptive = (flags & GEDWALK_ADAPTIVE_L) != 0;
  // One-step runs (directed graphs, lookahead off, spec_cols): phi^miss and the candidates likely to
  // win. One certifies most steps (a miss costs one candidate batch); on a directed graph the
  // adaptive variant certifies the best two exact gains, so it speculates on three.
  sh.cols_fused = adaptive && g.directed ? 4 : 2;
  if (r.spec_cols != 0) {
    if (!(r.spec_cols == 2 || r.spec_cols == 4 || (r.spec_cols == 8 && !r.fp64)))
      return fail(GEDWALK_ERR_INVALID, "spec_cols must be 0, 2, 4 or (FP32) 8");
    sh.cols_fused = r.spec_cols;
  }
  // Lookahead (undirected graphs): one run carries `levels` steps, level d under S + {c_1..c_d} with
  // the guessed winners c_d; a step whose winner was guessed needs no run of its own. The run's rows
  // hold levels + 1 columns. A gather costs one L2 sector request whatever the row width up to 32
  // bytes, so 7 FP32 levels (3 FP64) cost little more per sweep than one.
  const bool plain = (flags & (GEDWALK_ADAPTIVE_L | GEDWALK_STOCHASTIC | GEDWALK_GAINS_ALL)) == 0;
  sh.levels = 1;
  if (!g.directed && !(flags & GEDWALK_GAINS_ALL)) {
    sh.levels = r.fp64 ? 3 : 7;
    if (plain && r.lookahead != 0) {
      if (!(r.lookahead == 1 || r.lookahead == 3 || (!r.fp64 && r.lookahead == 7)))
        return fail(GEDWALK_ERR_INVALID, "lookahead must be 0, 1, 3 or (FP32) 7");
      sh.levels = r.lookahead;
    }
    if (!plain && r.spec_cols != 0) sh.levels = 1;  // the caller fixed the one-step width
  }
  // Candidate batches run when the evaluated guess is not certified: as wide as one sector carries
  // (undirected; directed batches hold no phi^miss column).
  sh.cols_cand = g.directed || r.fp64 ? 4 : 8;
  sh.cols_all = r.fp64 ? 8 : 16;
  sh.ell_max = 1;
  while (adaptive && sh.ell_max < r.L) sh.ell_max *= 2;
  sh.tab_L = adaptive ? sh.ell_max : r.L;
  sh.cols_max = std::max({sh.levels > 1 ? sh.levels + 1 : sh.cols_fused, sh.cols_cand,
                          (flags & GEDWALK_GAINS_ALL) ? sh.cols_all : 0, 2});
  *out = sh;
  return GEDWALK_OK;
}

int64_t maximize_footprint(const Graph& g, const Resolved& r, int32_t flags, int32_t k) {
  GreedyShape sh{};
  if (greedy_shape(g, r, flags, &sh) != GEDWALK_OK) return 0;
  const int64_t n = g.n, es = r.fp64 ? 8 : 4;
  if (!g.directed) {
    int64_t b = run_bytes(g, sh.tab_L, sh.cols_max, r.fp64, (flags & GEDWALK_GAINS_ALL) == 0);
    if ((flags & GEDWALK_GAINS_ALL) && small_gain_cols(g, r.fp64) > 0)  // one launch's table, vectors and gains
      b += n * (es * ((sh.tab_L + 1) / 2 + 3) + 8) + static_cast<int64_t>(std::max(g.plan.num_slots, 1)) * 8;
    return b + 4 * static_cast<int64_t>(k);  // (the final group, where it has to be scored)
  }
  const int64_t slices = std::max(std::max(g.plan.num_slices, g.plan_r.num_slices), 1);
  const int64_t heavy = std::max(std::max(g.plan.num_heavy, g.plan_r.num_heavy), 1);
  const int64_t slots = std::max(std::max(g.plan.num_slots, g.plan_r.num_slots), 1);
  int64_t b = 0;
  b += 2 * static_cast<int64_t>(sh.tab_L + 1) * n * es;  // phi^miss and psi^miss tables
  b += 2 * n * sh.cols_max * es;                         // walk vectors x0, x1
  b += slices * sh.cols_max * es + heavy * 4 + slots * sh.cols_max * 8 + sh.cols_max * kReduceParts * 8;
  b += (n + 31) / 32 * 4;                                // S bitmask
  b += n * static_cast<int64_t>(sizeof(Stale)) + static_cast<int64_t>(kSelBlocks) * kTopK * 8;
  b += static_cast<int64_t>(sizeof(SelOut)) + 16 * 4 + 16 * 8 + 256;
  return b;
}

namespace {
// What both loops need to know of a maximisation.
struct GreedyRun {
  int32_t k;
  int32_t flags;
  GreedyShape shape;
  double tol;       // relative inflation of bounds against rounding
  double eps_sep;   // adaptive: the separation
  double coef;      // adaptive: B_l = coef * Wa[l] (Eq. comb-bound, or Lemma spectral-bound)
  std::vector<double> Wa;
  double sample_m;  // stochastic: about this many vertices outside S are sampled per step (Appendix D)
  bool adaptive() const { return (flags & GEDWALK_ADAPTIVE_L) != 0; }
  bool stochastic() const { return (flags & GEDWALK_STOCHASTIC) != 0; }
  bool gains_all() const { return (flags & GEDWALK_GAINS_ALL) != 0; }
  double bound_at(int32_t l) const { return coef * Wa[l]; }
  // Step st's sample: vertex v (caller id) is drawn when hash(seed, st, v) < threshold, i.e. with
  // probability p = m / |V \ S|; UINT64_MAX: all of V \ S.
  uint64_t threshold(const Graph& g, int32_t st) const {
    if (stochastic() && st < g.n) {
      const double p = sample_m / static_cast<double>(g.n - st);
      const double scaled = p * 18446744073709551616.0;
      if (p < 1.0 && scaled < 18446744073709551615.0) return static_cast<uint64_t>(scaled);
    }
    return ~0ull;
  }
};

// Isolated vertices (rows [n_active, n)) start and end no walk: their bound and gain are exactly
// 0. The selections skip them, and the smallest caller id among those outside S stands for them
// among the zero gains. Stochastic greedy scans them all: they belong to its samples. The
// relabelling is a stable sort by degree, so the isolated rows hold increasing caller ids.
struct Isolated {
  int32_t next;
  unsigned long long zero(const Graph& g, const std::vector<char>& inS, unsigned long long z) {
    while (next < g.n && inS[next]) ++next;
    if (next < g.n)
      z = std::min(z, (static_cast<unsigned long long>(g.perm[next]) << 32) | static_cast<uint32_t>(next));
    return z;
  }
};

// The greedy loop of an undirected graph, on runs of half the walk length (run.cu).
gedwalk_status maximize_runs(Graph& g, Workspace& ws, const Resolved& r, const GreedyRun& p,
                             const std::vector<int32_t>& init, int32_t* group, double* gains,
                             std::vector<int32_t>* S_all) {
  const GreedyShape& sh = p.shape;
  const bool chain = sh.levels > 1;
  const int n_spec = chain ? sh.levels : sh.cols_fused - 1;
  const bool select = !p.gains_all();
  RunEngine eng(g, ws, r, r.stream);
  eng.n_scan = p.stochastic() ? g.n : g.n_active;
  eng.draws = p.stochastic();
  GW_TRY(eng.setup(sh.tab_L, sh.cols_max, select, init));
  GW_TRY(eng.set_length(p.adaptive() ? 1 : r.L, select));
  std::vector<char> inS(g.n, 0);
  for (int32_t v : init) inS[v] = 1;
  *S_all = init;
  Isolated iso{eng.n_scan};
  auto draws = [&](int32_t step) {
    eng.in->step = step;
    eng.in->seed = r.seed;
    for (int l = 0; l < kRunLevels; ++l) eng.in->thr[l] = p.threshold(g, step + l);
  };
  // Guesses from stored bounds: the best outside S, or per coming step the best of its sample.
  auto guess = [&](int32_t step, std::vector<int32_t>* to) -> gedwalk_status {
    draws(step);
    GW_TRY(eng.guess(p.stochastic() ? n_spec : 1));
    to->clear();
    for (int l = 0; l < n_spec; ++l) {
      const LevelSel& sel = eng.out->lv[p.stochastic() ? l : 0];
      int32_t pick = -1;
      for (int j = 0; j < kTopK && pick < 0; ++j)
        if (sel.id[j] != INT_MAX && std::find(to->begin(), to->end(), sel.id[j]) == to->end()) pick = sel.id[j];
      if (pick < 0) break;
      to->push_back(pick);
    }
    return GEDWALK_OK;
  };
  std::vector<int32_t> spec;
  if (select && p.k > 0) GW_TRY(guess(0, &spec));
  RunOut look{};                // the last run's answers, and
  std::vector<int32_t> look_c;  // its guesses
  int lvl = -1;                 // its level that stands under the current S (-1: none)

  for (int32_t step = 0; step < p.k; ++step) {
    Cand best{-1.0, -1, INT_MAX};
    if (p.gains_all()) {
      const unsigned long long z = iso.zero(g, inS, kNoZero);  // isolated vertices gain nothing
      if (z != kNoZero) best = Cand{0.0, zero_internal(z), zero_caller(z)};
      std::vector<int32_t> batch;
      const bool small = small_gain_cols(g, r.fp64) > 0;
      if (small) {
        std::vector<double> got(g.n_active);
        GW_TRY(small_gains(g, ws, r, *S_all, got.data()));
        for (int32_t v = 0; v < g.n_active; ++v) {
          if (inS[v]) continue;
          const Cand e{got[v], v, g.perm[v]};
          if (best.v < 0 || cand_before(e, best)) best = e;
          ++ws.st_evals;
        }
        ++ws.st_batches;
      }
      for (int32_t v = 0; !small && v <= g.n_active; ++v) {
        if (v < g.n_active && !inS[v]) batch.push_back(v);
        if (static_cast<int>(batch.size()) < sh.cols_all - 1 && !(v == g.n_active && !batch.empty())) continue;
        GW_TRY(eng.run(false, sh.cols_all, false, batch));
        for (size_t j = 0; j < batch.size(); ++j) {
          Cand e{eng.out->gains[j], batch[j], g.perm[batch[j]]};
          if (best.v < 0 || cand_before(e, best)) best = e;
        }
        ws.st_evals += static_cast<int64_t>(batch.size());
        ++ws.st_batches;
        batch.clear();
      }
    } else {
      for (;;) {  // one attempt per walk length (a single attempt unless adaptive)
        std::vector<Cand> E;  // evaluated with the current S
        if (lvl < 0) {
          look_c = spec;
          look_c.resize(n_spec, -1);
          draws(step);
          GW_TRY(eng.run(chain, n_spec + 1, true, look_c));
          look = *eng.out;
          lvl = 0;
          for (int32_t v : look_c) ws.st_evals += v >= 0;
          ++ws.st_batches;
        }
        LevelSel sel = look.lv[lvl];
        for (int j = chain ? lvl : 0; j < (chain ? lvl + 1 : n_spec); ++j)
          if (look_c[j] >= 0) E.push_back(Cand{look.gains[j], look_c[j], g.perm[look_c[j]]});
        const bool guessed = !E.empty();
        bool everyone = false;  // an empty sample: all of V \ S competes
        if (p.threshold(g, step) != ~0ull && sel.sampled == 0) {
          everyone = true;
          draws(step);
          eng.in->thr[0] = ~0ull;
          for (const Cand& e : E) eng.stale(e.v, e.g, step);
          GW_TRY(eng.run(false, sh.cols_cand, true, {}));
          sel = eng.out->lv[0];
        }
        bool first_batch = true, separated = true;
        std::vector<Cand> X;  // exact values for the current S, best first
        std::vector<int32_t> top;
        const int32_t left = g.n - static_cast<int32_t>(S_all->size());
        for (;;) {
          // certify: the best exact value beats every bound not yet evaluated (a zero bound is an
          // exact zero gain; the lowest such caller id stands for all of them)
          top.clear();
          for (int j = 0; j < kTopK; ++j)
            if (sel.id[j] != INT_MAX) top.push_back(sel.id[j]);
          X = E;
          const unsigned long long z = iso.zero(g, inS, sel.zero_min);
          if (z != kNoZero) X.push_back(Cand{0.0, zero_internal(z), zero_caller(z)});
          std::sort(X.begin(), X.end(), cand_before);
          const double ub0 = top.empty() ? -1.0 : static_cast<double>(sel.val[0]) * (1.0 + p.tol);
          const bool u_ok = top.empty() || (!X.empty() && ub0 < X[0].g);
          bool decided = u_ok;
          if (p.adaptive()) {
            // Separation test (Algorithm 2): u, the best, is taken when L(u) > L(v) + B_l - eps_sep,
            // v the best of the rest (a zero gain where nothing else is left to evaluate). The test
            // is monotone in L(u) and L(v), so bounds of them decide it wherever both of its
            // outcomes agree; the last vertex outside S needs no v.
            const double B = p.bound_at(eng.L);
            auto test = [&](double gu, double gv) { return gu > (gv + B) - p.eps_sep; };
            const double gu = X.empty() ? -1.0 : X[0].g;
            const double v_lo = X.size() >= 2 ? X[1].g : 0.0, v_hi = std::max(v_lo, ub0);
            if (left <= 1) {
              separated = true;
            } else if (!test(std::max(gu, ub0), 0.0)) {
              separated = false;  // even the best possible gain is not separated
              decided = true;
            } else if (u_ok) {
              separated = test(gu, v_hi);
              decided = separated || !test(gu, v_lo);
            }
          }
          if (decided) break;
          if (first_batch) {
            ws.st_spec_miss += guessed;
            for (const Cand& e : E) eng.stale(e.v, e.g, step);
          }
          first_batch = false;
          std::vector<int32_t> last(top.begin(), top.begin() + std::min<size_t>(top.size(), sh.cols_cand - 1));
          draws(step);
          if (everyone) eng.in->thr[0] = ~0ull;
          GW_TRY(eng.run(false, sh.cols_cand, true, last));
          for (size_t j = 0; j < last.size(); ++j) E.push_back(Cand{eng.out->gains[j], last[j], g.perm[last[j]]});
          ws.st_evals += static_cast<int64_t>(last.size());
          ++ws.st_batches;
          sel = eng.out->lv[0];
        }
        best = X.empty() ? Cand{-1.0, -1, INT_MAX} : X[0];
        // guesses for the next run: best remaining values, exact or not (a retry keeps the best too)
        std::vector<Cand> pool(X.begin() + (X.empty() || !separated ? 0 : 1), X.end());
        for (size_t j = 0; j < top.size(); ++j)
          pool.push_back(Cand{static_cast<double>(sel.val[j]), top[j], g.perm[top[j]]});
        std::sort(pool.begin(), pool.end(), cand_before);
        spec.clear();
        for (const Cand& e : pool)
          if (static_cast<int>(spec.size()) < n_spec && e.g > 0.0) spec.push_back(e.v);
        if (separated) break;
        ++ws.st_sep_fail;
        if (2 * eng.L > sh.ell_max)
          return fail(GEDWALK_ERR_DEVICE, "walk length passed %d without separation", sh.ell_max);
        // the bounds of the shorter length are no upper bounds for the longer one: reset them
        GW_TRY(eng.set_length(2 * eng.L, true));
        GW_CUDA(cudaMemsetAsync(ws.stale.p, 0xff, static_cast<size_t>(g.n) * sizeof(Stale), r.stream));
        lvl = -1;
      }
      // the next level is valid only when this step took the vertex it assumed
      if (chain && best.v == look_c[lvl] && lvl + 1 < sh.levels && look_c[lvl + 1] >= 0) ++lvl;
      else lvl = -1;
    }
    if (best.v < 0) return fail(GEDWALK_ERR_INVALID, "no vertex left to add");
    ws.st_ell.push_back(eng.L);
    group[step] = best.caller;
    gains[step] = best.g;
    inS[best.v] = 1;
    S_all->push_back(best.v);
    eng.added.push_back(best.v);
    if (best.g == 0.0 && !p.stochastic() && !p.adaptive()) {
      // every remaining gain is 0 (submodularity): the lowest caller ids follow
      int32_t caller = 0;
      while (++step < p.k) {
        while (inS[g.inv[caller]]) ++caller;
        const int32_t v = g.inv[caller];
        inS[v] = 1;
        S_all->push_back(v);
        ws.st_ell.push_back(eng.L);
        group[step] = caller;
        gains[step] = 0.0;
      }
      break;
    }
    if (p.stochastic() && lvl < 0 && step + 1 < p.k) GW_TRY(guess(step + 1, &spec));
  }
  ws.st_sweeps = eng.sweeps;
  return GEDWALK_OK;
}

// The greedy loop of a directed graph: one-step fused runs of the full length.
gedwalk_status maximize_directed(Graph& g, Workspace& ws, const Resolved& r, const GreedyRun& p,
                                 const std::vector<int32_t>& init_int, int32_t* group, double* gains,
                                 std::vector<int32_t>* S_out) {
  const int32_t k = p.k;
  cudaStream_t s = r.stream;
  const size_t es = r.fp64 ? 8 : 4;
  const bool adaptive = p.adaptive(), gains_all = p.gains_all(), stochastic = p.stochastic();
  const int cols_fused = p.shape.cols_fused, cols_cand = p.shape.cols_cand, cols_all = p.shape.cols_all;
  const int n_spec = cols_fused - 1;
  const double tol = p.tol;
  const int32_t ell_max = p.shape.ell_max;
  const int32_t L = p.shape.tab_L;  // rows of the miss table
  GW_TRY(ws.mtab.ensure(static_cast<size_t>(L + 1) * g.n * es, s));
  GW_TRY(zero_isolated_tail(g, ws.mtab.p, es, L, s));
  GW_TRY(ws.ztab.ensure(static_cast<size_t>(L + 1) * g.n * es, s));
  GW_TRY(zero_isolated_tail(g, ws.ztab.p, es, L, s));
  GW_TRY(ws.stale.ensure(static_cast<size_t>(g.n) * sizeof(Stale), s));
  GW_TRY(ws.sel.ensure(static_cast<size_t>(kSelBlocks) * kTopK * 8, s));
  GW_TRY(ws.small.ensure(sizeof(SelOut) + 16 * sizeof(int32_t) + 16 * sizeof(double) + 256, s));
  GW_TRY(ws.ensure_pinned(sizeof(SelOut) + 64));
  GW_TRY(upload_mask(g, ws, init_int, s));
  GW_CUDA(cudaMemsetAsync(ws.stale.p, 0xff, static_cast<size_t>(g.n) * sizeof(Stale), s));  // step -1, ub NaN

  GreedyCtx c{g, ws, r, s, adaptive ? 1 : r.L, es};
  const int need = adaptive ? 2 : 1;
  c.d_out = ws.small.as<SelOut>();
  c.d_cand = reinterpret_cast<int32_t*>(c.d_out + 1);
  c.d_gains = reinterpret_cast<double*>(c.d_cand + 16);
  c.h_out = static_cast<SelOut*>(ws.pinned);
  float* sel_v = ws.sel.as<float>();
  int* sel_id = reinterpret_cast<int*>(sel_v + kSelBlocks * kTopK);
  Stale* stale = ws.stale.as<Stale>();

  std::vector<uint32_t> hmask((static_cast<size_t>(g.n) + 31) / 32, 0u);
  std::vector<char> inS(g.n, 0);
  for (int32_t v : init_int) {
    hmask[v >> 5] |= 1u << (v & 31);
    inS[v] = 1;
  }
  std::vector<int32_t>& S_all = *S_out;
  S_all = init_int;
  std::vector<Cand> spec;  // next step's speculative candidates (internal ids)
  auto sampling_for = [&](int32_t st) { return Sampling{p.threshold(g, st), r.seed, static_cast<uint32_t>(st)}; };
  const int32_t n_scan = stochastic ? g.n : g.n_active;
  Isolated iso{n_scan};
  const int nb_sel = sel_blocks(n_scan);
  // One bound + selection pass into c.d_out / c.h_out; `step` decides which stale gains are exact.
  auto select_pass = [&](int32_t st, const Sampling& smp) -> gedwalk_status {
    reset_selection<<<1, 1, 0, s>>>(c.d_out);
    GW_KCHECK();
    if (r.fp64)
      GW_CUDA(launch_ub_select<double>(nb_sel, s, ws.mtab.as<double>(), ws.ztab.as<double>(), c.L, g.n, n_scan,
                                       ws.mask.as<uint32_t>(), stale, st, g.perm_d.as<int32_t>(), sel_v, sel_id, c.d_out,
                                       smp));
    else
      GW_CUDA(launch_ub_select<float>(nb_sel, s, ws.mtab.as<float>(), ws.ztab.as<float>(), c.L, g.n, n_scan,
                                      ws.mask.as<uint32_t>(), stale, st, g.perm_d.as<int32_t>(), sel_v, sel_id, c.d_out,
                                      smp));
    count_launch();
    GW_CUDA(cudaMemcpyAsync(c.h_out, c.d_out, sizeof(SelOut), cudaMemcpyDeviceToHost, s));
    GW_CUDA(cudaStreamSynchronize(s));
    read_graph_timing(ws);
    c.h_out->zero_min = iso.zero(g, inS, c.h_out->zero_min);
    return GEDWALK_OK;
  };

  for (int32_t step = 0; step < k; ++step) {
    std::vector<Cand> E;  // evaluated with the current S
    Cand best{-1.0, -1, INT_MAX};
    if (gains_all) {
      GW_TRY(run_sweeps(c, MODE_FUSED, 1, {}));
      std::vector<int32_t> batch;
      for (int32_t v = 0; v <= g.n; ++v) {
        if (v < g.n && !inS[v]) batch.push_back(v);
        if (static_cast<int>(batch.size()) == cols_all || (v == g.n && !batch.empty())) {
          GW_TRY(run_sweeps(c, MODE_CAND, cols_all, batch));
          double hg[16];
          GW_CUDA(cudaMemcpyAsync(hg, c.d_gains, sizeof(double) * cols_all, cudaMemcpyDeviceToHost, s));
          GW_CUDA(cudaStreamSynchronize(s));
          read_graph_timing(ws);
          for (size_t j = 0; j < batch.size(); ++j) {
            Cand e{hg[j], batch[j], g.perm[batch[j]]};
            if (best.v < 0 || cand_before(e, best)) best = e;
          }
          ws.st_evals += static_cast<int64_t>(batch.size());
          ++ws.st_batches;
          batch.clear();
        }
      }
    } else {
      Sampling smp = sampling_for(step);
      for (;;) {  // one attempt per walk length (a single attempt unless adaptive)
        // 1. psi^miss on the reverse CSR, then fused sweeps: phi^miss under S plus the speculative
        // candidates
        std::vector<int32_t> sc, last;
        E.clear();
        GW_TRY(run_sweeps(c, MODE_FUSED, 1, {}, true));
        for (const Cand& e : spec) sc.push_back(e.v);
        GW_TRY(run_sweeps(c, MODE_FUSED, sc.empty() ? 1 : cols_fused, sc));
        last = sc;
        bool first_batch = true;
        std::vector<Cand> X;  // exact values for the current S, best first
        std::vector<int32_t> top;
        for (;;) {
          if (!last.empty()) {
            update_stale<<<1, 32, 0, s>>>(stale, c.d_cand, c.d_gains, static_cast<int>(last.size()), step,
                                          c.d_out->gains);
            GW_KCHECK();
          }
          // 2. bound + selection pass
          GW_TRY(select_pass(step, smp));
          if (smp.thr != ~0ull && c.h_out->sampled == 0) {  // empty sample: all of V \ S competes
            smp.thr = ~0ull;
            continue;
          }
          for (size_t j = 0; j < last.size(); ++j) E.push_back(Cand{c.h_out->gains[j], last[j], g.perm[last[j]]});
          ws.st_evals += static_cast<int64_t>(last.size());
          if (!last.empty()) ++ws.st_batches;
          // 3. certify: the first `need` exact values beat every bound not yet evaluated (a zero
          // bound is an exact zero gain; the lowest such caller id stands for all of them)
          top.clear();
          for (int j = 0; j < kTopK; ++j)
            if (c.h_out->id[j] != INT_MAX) top.push_back(c.h_out->id[j]);
          X = E;
          const unsigned long long zmin = c.h_out->zero_min;
          if (zmin != kNoZero) X.push_back(Cand{0.0, zero_internal(zmin), zero_caller(zmin)});
          std::sort(X.begin(), X.end(), cand_before);
          const double ub0 = top.empty() ? -1.0 : static_cast<double>(c.h_out->val[0]) * (1.0 + tol);
          const bool certified =
              top.empty() || (static_cast<int>(X.size()) >= need && ub0 < X[need - 1].g);
          if (certified) break;
          if (first_batch && !sc.empty()) ++ws.st_spec_miss;
          first_batch = false;
          last.assign(top.begin(), top.begin() + std::min<size_t>(top.size(), cols_cand));
          GW_TRY(run_sweeps(c, MODE_CAND, cols_cand, last));
        }
        best = X.empty() ? Cand{-1.0, -1, INT_MAX} : X[0];
        // speculative candidates for the next step (or attempt): best remaining values, exact or not
        std::vector<Cand> pool(X.begin() + (X.empty() ? 0 : 1), X.end());
        for (size_t j = 0; j < top.size(); ++j)
          pool.push_back(Cand{static_cast<double>(c.h_out->val[j]), top[j], g.perm[top[j]]});
        std::sort(pool.begin(), pool.end(), cand_before);
        spec.clear();
        for (const Cand& e : pool) {
          if (static_cast<int>(spec.size()) == n_spec) break;
          if (e.g > 0.0) spec.push_back(e);
        }
        if (!adaptive) break;
        // separation test (Algorithm 2): u = best is taken when L(u) > U(v) - eps_sep, where v is
        // the best of the rest and U = L + B_l. With every other vertex unevaluated the rest has
        // zero gains; with u the last vertex outside S there is no v.
        const int32_t left = g.n - static_cast<int32_t>(S_all.size());
        const double gv = X.size() >= 2 ? X[1].g : 0.0;
        if (left <= 1 || best.g > (gv + p.bound_at(c.L)) - p.eps_sep) break;
        ++ws.st_sep_fail;
        if (2 * c.L > ell_max) return fail(GEDWALK_ERR_DEVICE, "walk length passed %d without separation", ell_max);
        c.L *= 2;
        // the bounds of the shorter length are no upper bounds for the longer one: reset them
        GW_CUDA(cudaMemsetAsync(ws.stale.p, 0xff, static_cast<size_t>(g.n) * sizeof(Stale), s));
        spec.clear();  // u and the runners-up are the best guesses at the longer length
        for (const Cand& e : X) {
          if (static_cast<int>(spec.size()) == n_spec) break;
          if (e.g > 0.0) spec.push_back(e);
        }
      }
    }
    ws.st_ell.push_back(c.L);
    if (best.v < 0) return fail(GEDWALK_ERR_INVALID, "no vertex left to add");
    group[step] = best.caller;
    gains[step] = best.g;
    const int32_t w = best.v;
    inS[w] = 1;
    S_all.push_back(w);
    hmask[w >> 5] |= 1u << (w & 31);
    GW_CUDA(cudaMemcpyAsync(ws.mask.as<uint32_t>() + (w >> 5), &hmask[w >> 5], 4, cudaMemcpyHostToDevice, s));
    spec.erase(std::remove_if(spec.begin(), spec.end(), [&](const Cand& e) { return e.v == w; }), spec.end());
    if (stochastic && step + 1 < k) {
      // The next step draws a new sample, so its speculative candidates are the best bounds
      // inside that sample: bounds and exact gains under the current S stay upper bounds once
      // w joins S (submodularity), which is all a speculative choice needs.
      spec.clear();
      const Sampling nxt = sampling_for(step + 1);
      GW_TRY(select_pass(step + 1, nxt));
      for (int j = 0; j < kTopK && static_cast<int>(spec.size()) < n_spec; ++j) {
        const int32_t id = c.h_out->id[j];
        if (id == INT_MAX || !(c.h_out->val[j] > 0.0f)) break;
        spec.push_back(Cand{static_cast<double>(c.h_out->val[j]), id, g.perm[id]});
      }
    }
  }
  ws.st_sweeps = c.sweeps;
  return GEDWALK_OK;
}

// Waits for a stream when a call leaves early with an error, so that nothing it launched still
// runs when its buffers are reused or freed.
struct SyncOnError {
  cudaStream_t s = nullptr;
  bool ok = false;
  ~SyncOnError() {
    if (!ok && s) {
      cudaStreamSynchronize(s);
      cudaGetLastError();
    }
  }
};
}  // namespace

gedwalk_status maximize_impl(Graph& g, Workspace& ws, int32_t k, const Resolved& r_in, int32_t flags,
                             const std::vector<int32_t>& init_int, int32_t* group, double* gains, double* score) {
  Resolved r = r_in;
  GW_TRY(greedy_stream(ws, r_in.stream, &r.stream));
  SyncOnError guard{r.stream};
  GreedyRun p{};
  p.k = k;
  p.flags = flags;
  GW_TRY(greedy_shape(g, r, flags, &p.shape));
  // Rounding of the values a certification compares, beyond what the bounds themselves allow for. A
  // run's first vector is exact counts and its sums are rounded a few times each (about 2e-7 in all,
  // measured against 64 bits); the full-length sweeps of a directed graph round more often.
  p.tol = r.fp64 ? 1e-11 : g.directed ? 1e-5 : 1e-6;
  if (p.stochastic() && (p.gains_all() || !init_int.empty()))
    return fail(GEDWALK_ERR_INVALID, "stochastic greedy cannot be combined with GEDWALK_GAINS_ALL or an init group");
  if (p.stochastic() && !(r.eta > 0.0 && r.eta < 1.0)) return fail(GEDWALK_ERR_INVALID, "eta must lie in (0, 1)");
  if (p.adaptive() && (p.gains_all() || p.stochastic() || !init_int.empty()))
    return fail(GEDWALK_ERR_INVALID,
                "GEDWALK_ADAPTIVE_L cannot be combined with GEDWALK_GAINS_ALL, GEDWALK_STOCHASTIC or an init group");
  if (p.adaptive() && !(r.eps > 0.0)) return fail(GEDWALK_ERR_INVALID, "GEDWALK_ADAPTIVE_L needs epsilon (L must be 0)");
  p.sample_m = std::ceil(static_cast<double>(g.n) / std::max(k, 1) * std::log(1.0 / (p.stochastic() ? r.eta : 0.5)));
  // adaptive: l runs through the powers of two from 1; B_l < eps_sep separates any pair, and r.L
  // (the first l with B_l < eps_sep) bounds the largest power reached.
  p.eps_sep = r.eps;
  if (p.adaptive()) {
    GW_TRY(bound_coef(g, r.alpha, r.bound_kind, r.stream, &p.coef));
    GW_TRY(ensure_totals(g, r.alpha, p.shape.ell_max + 1, r.stream));
    std::shared_lock<std::shared_mutex> rl(g.tt_lock);
    if (g.tt_alpha != r.alpha || g.tt_rows < p.shape.ell_max + 1)
      return fail(GEDWALK_ERR_INVALID, "the walk-total table was replaced for another alpha during the call");
    p.Wa.assign(g.Wa.begin(), g.Wa.begin() + p.shape.ell_max + 1);
  }
  ws.st_evals = ws.st_batches = ws.st_sweeps = ws.st_spec_miss = ws.st_sep_fail = 0;
  ws.st_ell.clear();
  std::vector<int32_t> S_all;
  if (g.directed) GW_TRY(maximize_directed(g, ws, r, p, init_int, group, gains, &S_all));
  else GW_TRY(maximize_runs(g, ws, r, p, init_int, group, gains, &S_all));
  if (score) {
    // GED_{<=L} of the final group. From an empty start it is the sum of the picks' exact gains
    // g_L(S_j, c_j) = GED_{<=L}(S_j + c_j) - GED_{<=L}(S_j), telescoping from GED_{<=L}(empty) = 0;
    // otherwise (an init group, or gains at shorter walk lengths) the group is scored.
    if (init_int.empty() && !p.adaptive()) {
      double v = 0.0;
      for (int32_t j = 0; j < k; ++j) v += gains[j];
      *score = v;
    } else {
      GW_TRY(score_one(g, ws, S_all, r, score));
    }
  }
  GW_CUDA(cudaStreamSynchronize(r.stream));
  guard.ok = true;
  return GEDWALK_OK;
}

gedwalk_status gains_impl(Graph& g, Workspace& ws, const std::vector<int32_t>& S_int, const Resolved& r_in,
                          double* gains_caller) {
  Resolved r = r_in;
  GW_TRY(greedy_stream(ws, r_in.stream, &r.stream));
  SyncOnError guard{r.stream};
  cudaStream_t s = r.stream;
  const size_t es = r.fp64 ? 8 : 4;
  const int cols_all = r.fp64 ? 8 : 16;
  std::vector<char> inS(g.n, 0);
  for (int32_t v : S_int) inS[v] = 1;
  for (int32_t v = 0; v < g.n; ++v) gains_caller[v] = 0.0;
  std::vector<int32_t> batch;
  if (small_gain_cols(g, r.fp64) > 0) {
    std::vector<double> got(g.n_active);
    GW_TRY(small_gains(g, ws, r, S_int, got.data()));
    for (int32_t v = 0; v < g.n_active; ++v) gains_caller[g.perm[v]] = got[v];
    guard.ok = true;
    return GEDWALK_OK;
  }
  if (!g.directed) {  // an isolated vertex gains nothing
    RunEngine eng(g, ws, r, s);
    GW_TRY(eng.setup(r.L, cols_all, false, S_int));
    GW_TRY(eng.set_length(r.L, false));
    for (int32_t v = 0; v <= g.n_active; ++v) {
      if (v < g.n_active && !inS[v]) batch.push_back(v);
      if (static_cast<int>(batch.size()) < cols_all - 1 && !(v == g.n_active && !batch.empty())) continue;
      GW_TRY(eng.run(false, cols_all, false, batch));
      for (size_t j = 0; j < batch.size(); ++j) gains_caller[g.perm[batch[j]]] = eng.out->gains[j];
      batch.clear();
    }
    GW_CUDA(cudaStreamSynchronize(s));
    guard.ok = true;
    return GEDWALK_OK;
  }
  GW_TRY(ws.mtab.ensure(static_cast<size_t>(r.L + 1) * g.n * es, s));
  GW_TRY(zero_isolated_tail(g, ws.mtab.p, es, r.L, s));
  GW_TRY(ws.small.ensure(sizeof(SelOut) + 16 * sizeof(int32_t) + 16 * sizeof(double) + 256, s));
  GW_TRY(upload_mask(g, ws, S_int, s));
  GreedyCtx c{g, ws, r, s, r.L, es};
  c.d_out = ws.small.as<SelOut>();
  c.d_cand = reinterpret_cast<int32_t*>(c.d_out + 1);
  c.d_gains = reinterpret_cast<double*>(c.d_cand + 16);
  GW_TRY(run_sweeps(c, MODE_FUSED, 1, {}));
  for (int32_t v = 0; v <= g.n; ++v) {
    if (v < g.n && !inS[v]) batch.push_back(v);
    if (static_cast<int>(batch.size()) == cols_all || (v == g.n && !batch.empty())) {
      GW_TRY(run_sweeps(c, MODE_CAND, cols_all, batch));
      double hg[16];
      GW_CUDA(cudaMemcpyAsync(hg, c.d_gains, sizeof(double) * cols_all, cudaMemcpyDeviceToHost, s));
      GW_CUDA(cudaStreamSynchronize(s));
      read_graph_timing(ws);
      for (size_t j = 0; j < batch.size(); ++j) gains_caller[g.perm[batch[j]]] = hg[j];
      batch.clear();
    }
  }
  guard.ok = true;
  return GEDWALK_OK;
}

}  // namespace gw

using namespace gw;

extern "C" {

gedwalk_status gedwalk_maximize(gedwalk_graph_t h, int32_t k, const gedwalk_params* params, int32_t* group,
                                double* gains, double* score, int32_t* L_used, const int32_t* init_group,
                                int32_t init_len) {
  if (!h) return fail(GEDWALK_ERR_INVALID, "graph is NULL");
  if (k < 0) return fail(GEDWALK_ERR_INVALID, "k must be >= 0");
  if (k > 0 && !group) return fail(GEDWALK_ERR_INVALID, "group is NULL");
  Graph* g = G(h);
  std::lock_guard<std::mutex> lk(g->mu);
  GW_CUDA(cudaSetDevice(g->device));
  std::vector<int32_t> init;
  GW_TRY(map_group(*g, init_group, init_len, &init));
  if (static_cast<int64_t>(init.size()) + k > g->n)
    return fail(GEDWALK_ERR_INVALID, "init group (%zu) + k (%d) exceeds n (%d)", init.size(), k, g->n);
  gedwalk_params d;
  gedwalk_params_default(&d);
  const gedwalk_params* p = params ? params : &d;
  const double eps = (p->greedy_eps_rule == GEDWALK_EPS_OVER_K && k > 0) ? p->epsilon / k : p->epsilon;
  Resolved r;
  GW_TRY(resolve(*g, p, eps, &r));
  std::vector<int32_t> grp(std::max(k, 1));
  std::vector<double> gn(std::max(k, 1));
  double sc = 0;
  GW_TRY(maximize_impl(*g, g->ws, k, r, p->flags, init, grp.data(), gn.data(), score ? &sc : nullptr));
  g->st_evals = g->ws.st_evals;
  g->st_batches = g->ws.st_batches;
  g->st_sweeps = g->ws.st_sweeps;
  g->st_spec_miss = g->ws.st_spec_miss;
  g->st_ell = g->ws.st_ell;
  g->st_sep_fail = g->ws.st_sep_fail;
  for (int32_t j = 0; j < k; ++j) {
    group[j] = grp[j];
    if (gains) gains[j] = gn[j];
  }
  if (score) *score = sc;
  if (L_used) *L_used = (p->flags & GEDWALK_ADAPTIVE_L) ? (g->st_ell.empty() ? 1 : g->st_ell.back()) : r.L;
  return GEDWALK_OK;
}

gedwalk_status gedwalk_maximize_lengths(gedwalk_graph_t h, int32_t* ell, int32_t cap, int32_t* count,
                                        int64_t* separation_failures) {
  if (!h) return fail(GEDWALK_ERR_INVALID, "graph is NULL");
  if (cap < 0 || (cap > 0 && !ell)) return fail(GEDWALK_ERR_INVALID, "ell is NULL or cap < 0");
  Graph* g = G(h);
  std::lock_guard<std::mutex> lk(g->mu);
  const int32_t m = static_cast<int32_t>(g->st_ell.size());
  for (int32_t j = 0; j < std::min(m, cap); ++j) ell[j] = g->st_ell[j];
  if (count) *count = m;
  if (separation_failures) *separation_failures = g->st_sep_fail;
  return GEDWALK_OK;
}

gedwalk_status gedwalk_maximize_stats(gedwalk_graph_t h, int64_t* evaluations, int64_t* batches, int64_t* sweeps,
                                      int64_t* spec_misses) {
  if (!h) return fail(GEDWALK_ERR_INVALID, "graph is NULL");
  Graph* g = G(h);
  std::lock_guard<std::mutex> lk(g->mu);
  if (evaluations) *evaluations = g->st_evals;
  if (batches) *batches = g->st_batches;
  if (sweeps) *sweeps = g->st_sweeps;
  if (spec_misses) *spec_misses = g->st_spec_miss;
  return GEDWALK_OK;
}

gedwalk_status gedwalk_gains(gedwalk_graph_t h, const int32_t* S, int32_t s_len, const gedwalk_params* params,
                             double* gains, int32_t* L_used) {
  if (!h || !gains) return fail(GEDWALK_ERR_INVALID, "graph or gains is NULL");
  Graph* g = G(h);
  std::lock_guard<std::mutex> lk(g->mu);
  GW_CUDA(cudaSetDevice(g->device));
  std::vector<int32_t> S_int;
  GW_TRY(map_group(*g, S, s_len, &S_int));
  Resolved r;
  GW_TRY(resolve(*g, params, 0.0, &r));
  GW_TRY(gains_impl(*g, g->ws, S_int, r, gains));
  if (L_used) *L_used = r.L;
  return GEDWALK_OK;
}

}  // extern "C"
