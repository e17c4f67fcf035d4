// Runs of the greedy maximisation: sweeps of half the walk length and the pass in which the halves
// meet.
//
// With M = alpha 1_{V\S} A symmetric on V \ S, a walk of length a + b that avoids S is a walk of
// length a and one of length b that end at the same vertex v (its vertex number a). So with
// phi_t(v) the S-avoiding walks of length t that end at v, and k_t(v) those among them that visit
// c, the walks of length a + b through c number
//     sum_v [ k_a(v) phi_b(v) + (phi_a(v) - k_a(v)) k_b(v) ]
// (the first half visits c, or it does not and the second half does). All terms are >= 0. The gain
// of c sums the lengths 1..L; with H = ceil(L/2), the lengths up to H are plain sums of k_t and
// every length H + a, a = 1..L-H, pairs with b = H:
//     gain(c) = sum_v [ K(v) + V(v) phi_H(v) + (P(v) - V(v)) k_H(v) ],
//     K = sum_{t=1..H} k_t,  V = sum_{t=1..L-H} k_t,  P = sum_{t=1..L-H} phi_t.
// Half the sweeps, one pass over the stored vectors. Weighted graphs (symmetric weights) alike.
//
// The first sweep is no sweep either: phi_1(v) = alpha |N(v) \ S| is a count kept per vertex, and
// k_1 is alpha on the candidate's neighbours. (Weighted graphs sweep from the unit vectors.)
//
// Directed graphs keep two sets of vectors: walks that start at v (sweeps along the given rows) and
// walks that end at v (sweeps along the reverse CSR). A walk of length H + a is a walk of length a
// that ends at v and one of length H that starts there, so with the starting walks phi, k and the
// ending walks psi, j:  gain(c) = sum_v [ K(v) + V(v) phi_H(v) + (P(v) - V(v)) k_H(v) ] with V and P
// summed over j and psi. As many sweeps as the full length in one orientation, for up to seven steps.
//
// Bounds. The gain pairs first visits with continuations, sum_{1<=p+q<=L} f_p phi_q at c, where
// f_p <= phi_p counts the walks whose only visit to c is their end: f_p = phi_p - sum_m s_m phi_{p-m}
// with s_m the closed walks from c that return first at step m. Any lower bounds of s_m give an
// upper bound of f: s_2 = alpha^2 |N(c) \ S| exactly, s_4 >= alpha^2 phi_2 - alpha^3 phi_1 (c-u-v-u-c,
// v != c). With p, q <= H all pairs but (0,0) (and, for odd L, (H,H)) belong to the sum, so it is
// F + U + F U with U = sum phi_t, F = sum f_t: no convolution. The pairs with p or q above H are
// bounded once per maximisation by their value without S (walks avoiding S only get fewer as S
// grows), from the walk-total tables. (Directed: F sums psi, U phi; the returns are not counted.)
//
// Measured on a GB300 (one maximisation, before: full-length sweeps that store every level's phi, a
// bound pass per step and the visits-times-continuations bound): R-MAT scale 22, k = 100, FP32 126 to 144
// -> 33.6 to 38 ms, by the graph's seed (60 to 68 sweeps of 494 us instead of 135 of 587 and 54 of 498); Erdos-Renyi
// n = 100,003, degree 16, k = 27 18.1 -> 2.1 ms (the sharper bound leaves one or two candidate batches);
// Barabasi-Albert n = 10^6, k = 25, FP64 39.2 -> 7.5 ms (10.2 where a chain breaks); Algorithm 2 on R-MAT
// scale 20, k = 50 96.5 -> 10.1 ms.
#include <algorithm>
#include <cmath>

#include "run.h"

namespace gw {

uint64_t mix_all(std::initializer_list<uint64_t> vs) {
  uint64_t key = 0;
  for (uint64_t v : vs) key ^= v + 0x9e3779b97f4a7c15ULL + (key << 6) + (key >> 2);
  return key ? key : 1;  // 0 marks a free cache entry
}

gedwalk_status run_sequence(Workspace& ws, cudaStream_t s, const Sequence& q,
                            const std::function<gedwalk_status(bool, const std::vector<cudaEvent_t>*)>& issue) {
  if (s == nullptr) return issue(true, nullptr);
  // the workspace's entry for this configuration, else the least recently used one
  SweepGraph* hit = nullptr;
  SweepGraph* lru = &ws.graphs[0];
  for (SweepGraph& e : ws.graphs) {
    if (e.key == q.key) hit = &e;
    if (e.last_use < lru->last_use) lru = &e;
  }
  if (!hit) {
    lru->reset();
    lru->key = q.key;
    hit = lru;
  }
  SweepGraph& sg = *hit;
  sg.last_use = ++ws.graph_clock;
  if (!sg.exec) {
    if (sg.uses++ < (q.nnz > kLateEntries ? 3 : 1)) return issue(true, nullptr);  // set-up happens outside capture
    sg.ev.assign(2, nullptr);
    for (cudaEvent_t& e : sg.ev) GW_CUDA(cudaEventCreate(&e));
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();  // a stream that cannot be captured: directly, as ever
      sg.reset();
      return issue(true, nullptr);
    }
    set_capturing(true);
    const gedwalk_status st = issue(false, &sg.ev);
    set_capturing(false);
    cudaGraph_t graph = nullptr;
    const cudaError_t ce = cudaStreamEndCapture(s, &graph);
    if (st != GEDWALK_OK || ce != cudaSuccess || !graph) {
      // Nothing captured has run. Another thread can invalidate a capture (a call that waits for
      // the whole device, such as cudaFree); the sequence then runs directly, and a genuine error
      // shows up again there.
      if (graph) cudaGraphDestroy(graph);
      cudaGetLastError();
      sg.reset();
      return issue(true, nullptr);
    }
    const cudaError_t ie = cudaGraphInstantiate(&sg.exec, graph, 0);
    cudaGraphDestroy(graph);
    if (ie != cudaSuccess) {
      sg.exec = nullptr;
      sg.reset();
      return fail(GEDWALK_ERR_DEVICE, "graph instantiation failed: %s", cudaGetErrorString(ie));
    }
    sg.kernels = q.kernels;
    sg.sweeps = q.sweeps;
    sg.bytes = q.bytes;
    sg.prof_key = q.prof_key;
  }
  GW_CUDA(cudaGraphLaunch(sg.exec, s));
  count_launches(sg.kernels);
  sg.timing_pending = profiling();
  return GEDWALK_OK;
}

// The stream a run uses: the caller's, or (for the legacy default stream, handle 0 or cudaStreamLegacy,
// which cannot be captured) the workspace's own stream, ordered after the caller's.
gedwalk_status greedy_stream(Workspace& ws, cudaStream_t caller, cudaStream_t* out) {
  if (caller != nullptr && caller != cudaStreamLegacy) {
    *out = caller;
    return GEDWALK_OK;
  }
  if (!ws.own_stream) GW_CUDA(cudaStreamCreateWithFlags(&ws.own_stream, cudaStreamNonBlocking));
  if (!ws.order_ev) GW_CUDA(cudaEventCreateWithFlags(&ws.order_ev, cudaEventDisableTiming));
  GW_CUDA(cudaEventRecord(ws.order_ev, caller));
  GW_CUDA(cudaStreamWaitEvent(ws.own_stream, ws.order_ev, 0));
  *out = ws.own_stream;
  return GEDWALK_OK;
}

void read_graph_timing(Workspace& ws) {
  for (SweepGraph& sg : ws.graphs) {
    if (!sg.timing_pending) continue;
    sg.timing_pending = false;
    float ms = 0.0f;  // the run of sweeps, shared evenly among them
    if (sg.sweeps > 0 && sg.ev.size() == 2 && cudaEventElapsedTime(&ms, sg.ev[0], sg.ev[1]) == cudaSuccess) {
      for (int t = 0; t < sg.sweeps; ++t) profile_add(ms / sg.sweeps, sg.bytes, sg.prof_key);
    } else {
      cudaGetLastError();
    }
  }
}

namespace {

constexpr int kChunks = 32;  // blocks that share one vertex's neighbours (hubs have 10^5)

__device__ __forceinline__ bool in_set(const uint32_t* __restrict__ mask, int32_t v) {
  return (__ldg(mask + (v >> 5)) >> (v & 31)) & 1u;
}

// A graph's lists as the runs use them. o = 0: walks that start at a vertex, along its own row; o = 1
// (directed): walks that end there, along its row of the reverse CSR. cnt[o][v] = |row o of v cap S|.
struct Rows {
  const int32_t* rp[2];
  const int32_t* ci[2];
  int32_t* cnt[2];
  int directed;
};

// S grows by list[0..count): the mask bits, and the counts of every vertex whose row holds one of them.
__device__ __forceinline__ void join_set(const int32_t* __restrict__ list, int32_t count, const Rows& g,
                                         uint32_t* __restrict__ mask) {
  for (int32_t i = blockIdx.y; i < count; i += gridDim.y) {
    const int32_t v = list[i];
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(mask + (v >> 5), 1u << (v & 31));
    for (int o = 0; o <= g.directed; ++o) {
      const int r = g.directed ? 1 - o : 0;  // v is in row o of u where u is in v's other row
      const int64_t e1 = g.rp[r][v + 1];
      for (int64_t j = g.rp[r][v] + static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; j < e1;
           j += static_cast<int64_t>(gridDim.x) * blockDim.x)
        atomicAdd(g.cnt[o] + g.ci[r][j], 1);
    }
  }
}

// The same for a whole group, which may be half of the graph. With blockIdx.y = 0 a warp takes a member at a
// time and up to kJoinRow entries of its row; the other slices of the grid (where rows are longer than that)
// look through up to 32 members at a time for the rest of hubs' rows, which they share. A block per member
// took 30 ms for half of R-MAT scale 20, the sweeps 0.35. count: list[-1] when negative (a captured launch).
constexpr int kJoinRow = 256;
__global__ void join_kernel(const int32_t* __restrict__ list, int32_t count, const Rows g, uint32_t* __restrict__ mask) {
  if (count < 0) count = list[-1];
  const int lane = threadIdx.x & 31;
  const int32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, warps = (gridDim.x * blockDim.x) >> 5;
  if (blockIdx.y == 0) {
    for (int32_t i = warp; i < count; i += warps) {
      const int32_t v = list[i];
      if (lane == 0) atomicOr(mask + (v >> 5), 1u << (v & 31));
      for (int o = 0; o <= g.directed; ++o) {
        const int r = g.directed ? 1 - o : 0;  // v is in row o of u where u is in v's other row
        const int64_t e0 = g.rp[r][v], e1 = min(static_cast<int64_t>(g.rp[r][v + 1]), e0 + kJoinRow);
        for (int64_t e = e0 + lane; e < e1; e += 32) atomicAdd(g.cnt[o] + g.ci[r][e], 1);
      }
    }
    return;
  }
  const int slice = static_cast<int>(blockIdx.y) - 1, slices = static_cast<int>(gridDim.y) - 1;
  const int per = max(1, min(32, (count + warps - 1) / warps));  // few members: each its own warps
  for (int64_t i0 = per * static_cast<int64_t>(warp); i0 < count; i0 += per * static_cast<int64_t>(warps)) {
    const int32_t mine = lane < per && i0 + lane < count ? list[i0 + lane] : -1;
    for (int o = 0; o <= g.directed; ++o) {
      const int r = g.directed ? 1 - o : 0;
      const bool hub = mine >= 0 && g.rp[r][mine + 1] - g.rp[r][mine] > kJoinRow;
      for (unsigned m = __ballot_sync(kFullMask, hub); m; m &= m - 1) {
        const int32_t v = __shfl_sync(kFullMask, mine, __ffs(m) - 1);
        const int64_t e1 = g.rp[r][v + 1];
#pragma unroll 4
        for (int64_t e = static_cast<int64_t>(g.rp[r][v]) + kJoinRow + slice * 32 + lane; e < e1; e += 32 * slices)
          atomicAdd(g.cnt[o] + g.ci[r][e], 1);
      }
    }
  }
}

// Opens a run: the vertices that joined S, the exact gains known on the host, the pass's counters.
__global__ void run_begin(RunDev* __restrict__ d, const Rows g, uint32_t* __restrict__ mask, Stale* __restrict__ stale) {
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    const int t = threadIdx.x;
    if (t < 2 * kRunCols) d->adj[t / kRunCols][t % kRunCols] = 0;
    if (t < kRunLevels) {
      d->out.lv[t].zero_min = kNoZero;
      d->out.lv[t].sampled = 0;
    }
    if (t == 0) {
      d->done = 0;
      if (stale)
        for (int j = 0; j < d->in.n_stale; ++j)  // in order: a vertex may come twice
          stale[d->in.stale_id[j]] = Stale{__double2float_ru(d->in.stale_gain[j]), d->in.stale_step[j]};
    }
  }
  join_set(d->in.added, d->in.n_added, g, mask);
}

template <typename T>
struct Chunk16;
template <>
struct Chunk16<float> {
  using type = float4;
  __device__ static float4 make(const float* e) { return make_float4(e[0], e[1], e[2], e[3]); }
};
template <>
struct Chunk16<double> {
  using type = double2;
  __device__ static double2 make(const double* e) { return make_double2(e[0], e[1]); }
};

// The first stored vector of a run, rows [0, n_active). Unweighted: x_1, column 0 = alpha |N(v) \ S|
// (0 on S), the candidate columns 0 (run_scatter fills them). Weighted (rs): x_0 scaled by s, column
// 0 = s on V \ S, candidate column j = s at the candidate. 16 bytes per thread, consecutive.
template <typename T, int C>
__global__ void run_init(T* __restrict__ X, const RunDev* __restrict__ d, const int32_t* __restrict__ rp,
                         const int32_t* __restrict__ cnt, const uint32_t* __restrict__ mask, int32_t n_active, T alpha,
                         const T* __restrict__ rs) {
  constexpr int per = 16 / static_cast<int>(sizeof(T)) < C ? 16 / static_cast<int>(sizeof(T)) : C;
  constexpr int cpr = C / per;  // chunks per row
  const int64_t chunks = static_cast<int64_t>(n_active) * cpr;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; q < chunks; q += stride) {
    const int32_t v = static_cast<int32_t>(q / cpr);
    const int part = static_cast<int>(q % cpr);
    T e[per];
#pragma unroll
    for (int j = 0; j < per; ++j) e[j] = T(0);
    if (rs) {
      const T sv = rs[v];
      if (part == 0 && !in_set(mask, v)) e[0] = sv;
#pragma unroll
      for (int j = 0; j < per; ++j) {
        const int col = part * per + j;
        if (col > 0 && __ldg(&d->in.cand[col - 1]) == v) e[j] = sv;
      }
    } else if (part == 0 && !in_set(mask, v)) {
      e[0] = alpha * static_cast<T>(rp[v + 1] - rp[v] - cnt[v]);
    }
    if constexpr (per * sizeof(T) == 16) {
      reinterpret_cast<typename Chunk16<T>::type*>(X)[q] = Chunk16<T>::make(e);
    } else {
#pragma unroll
      for (int j = 0; j < per; ++j) X[q * per + j] = e[j];
    }
  }
}

// Unweighted x_1 of the candidate columns, one set of vectors per grid.z: alpha on the vertices whose
// row holds the candidate and which lie outside the column's base set (S, with the earlier candidates
// in a chain), and, for a chain, the number of earlier candidates in each candidate's row (found in
// its other row's scan on a directed graph). Weighted graphs take only the counts.
template <typename T, bool CHAIN>
__global__ void run_scatter(T* __restrict__ X, int64_t set, int cols, RunDev* __restrict__ d, const Rows g,
                            const uint32_t* __restrict__ mask, T alpha, int write) {
  __shared__ int sc[kRunCols];
  if (threadIdx.x < kRunCols) sc[threadIdx.x] = d->in.cand[threadIdx.x];
  __syncthreads();
  const int j = blockIdx.y, o = blockIdx.z, r = g.directed ? 1 - o : 0;
  const int32_t c = sc[j];
  if (c < 0) return;
  X += set * o;
  const int64_t e1 = g.rp[r][c + 1];
  for (int64_t e = g.rp[r][c] + static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; e < e1;
       e += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int32_t v = g.ci[r][e];
    bool base = false;
    if (CHAIN)
      for (int i = 0; i < j; ++i) base |= sc[i] == v;
    if (base) atomicAdd(&d->adj[r][j], 1);
    else if (write && !in_set(mask, v)) X[static_cast<size_t>(v) * cols + j + 1] = alpha;
  }
}

// The candidates' own rows: live[o][j] says whether c_j's row o has an entry outside its base set; x_1
// there is phi_1 under that set.
template <typename T, bool CHAIN>
__global__ void run_own(T* __restrict__ X, int64_t set, int cols, RunDev* __restrict__ d, const Rows g, T alpha, int write) {
  const int j = threadIdx.x, o = blockIdx.x;
  if (j >= kRunCols) return;
  const int32_t c = j < cols - 1 ? d->in.cand[j] : -1;
  int32_t dg = 0;
  if (c >= 0) {
    dg = g.rp[o][c + 1] - g.rp[o][c] - g.cnt[o][c] - (CHAIN ? d->adj[o][j] : 0);
    if (write) X[set * o + static_cast<size_t>(c) * cols + j + 1] = alpha * static_cast<T>(dg);
  }
  d->live[o][j] = dg > 0;
}

// Tail bounds from tables of walk totals (rows n apart; times s on a weighted graph): the pairs p + q <= L
// with p or q above H.
// A: walks that start at v, B: that end there, both to L (the same on an undirected graph):
//   tail(v) = sum_{p>H} b_p Qa_{L-p} + sum_{q>H} a_q Qb_{L-q},  Q_q = t_0 + ... + t_q.
// With M, an undirected graph's table of rows 0..H: t_{H+b}(v) <= t_H(v) M_b, M_b the largest t_b (a walk of
// length H + b from v is one of length H and one of length b from its end), so
//   tail(v) = 2 t_H(v) sum_{b=1..L-H} M_b Q_{L-H-b}.
// Rounded up, times `grow` for the table's own rounding; and (about) the bound of the empty group,
// F + U + F U + tail, for the first guesses.
__global__ void row_max_kernel(const double* __restrict__ A, int64_t n, int32_t n_active, const double* __restrict__ rs,
                               unsigned long long* __restrict__ M) {
  const double* row = A + static_cast<size_t>(blockIdx.y + 1) * n;
  double m = 0.0;
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n_active; v += gridDim.x * blockDim.x)
    m = fmax(m, rs ? row[v] / rs[v] : row[v]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(kFullMask, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(M + blockIdx.y + 1, static_cast<unsigned long long>(__double_as_longlong(m)));
}

template <typename T>
__global__ void tail_kernel(const T* __restrict__ A, const T* __restrict__ B, const double* __restrict__ M,
                            int64_t n, int32_t n_active, int32_t L, int32_t H, const T* __restrict__ rs, double alpha,
                            double grow, float* __restrict__ tail, float* __restrict__ bound) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n_active; v += gridDim.x * blockDim.x) {
    const double inv = rs ? 1.0 / rs[v] : 1.0;
    auto a = [&](int32_t t) { return A[static_cast<size_t>(t) * n + v] * inv; };
    auto b = [&](int32_t t) { return B[static_cast<size_t>(t) * n + v] * inv; };
    double Qa = 0.0, Qb = 0.0, acc = 0.0, U = 0.0, F = 0.0;
    if (M) {
      for (int32_t q = 0; q < L - H; ++q) {
        const double t = a(q);
        Qa += t;
        if (q > 0) U += t;
        acc += __ldg(M + (L - H - q)) * Qa;
      }
      for (int32_t t = std::max(L - H, 1); t < H; ++t) U += a(t);
      const double tH = a(H);
      U += tH;
      acc *= 2.0 * tH;
      const double f1 = a(1), f2 = H >= 2 ? a(2) : 0.0;
      const double s2 = rs ? 0.0 : alpha * f1, s4 = rs || H < 4 ? 0.0 : alpha * alpha * f2 - alpha * alpha * alpha * f1;
      F = U - (H >= 2 ? (s2 + s4) * (1.0 + U) : 0.0);
    } else {
      for (int32_t q = 0; q < L - H; ++q) {
        Qa += a(q);
        Qb += b(q);
        acc += b(L - q) * Qa + a(L - q) * Qb;
      }
      for (int32_t t = 1; t <= H; ++t) {
        U += a(t);
        F += b(t);
      }
    }
    acc *= grow;
    tail[v] = __double2float_ru(acc);
    bound[v] = static_cast<float>(F + U + F * U + acc);
  }
}

// Row 0 of a call's own table: 1 outside S (times s).
template <typename T>
__global__ void own_row0(T* __restrict__ row, const uint32_t* __restrict__ mask, int32_t n_active, const T* __restrict__ rs) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n_active; v += gridDim.x * blockDim.x)
    row[v] = in_set(mask, v) ? T(0) : rs ? rs[v] : T(1);
}

struct MeetArgs {
  const void* xs;      // x_1 .. x_H, each [n_active][C]
  const void* xr;      // directed: the same of the walks that end at a vertex
  int64_t stride;      // elements from x_t to x_{t+1}
  int32_t L, H;
  int32_t n_scan, n_active;
  Rows g;
  const uint32_t* mask;
  const int32_t* perm;
  const float* tail;
  float* bound;        // stochastic greedy: the last level's bounds (else nullptr)
  Stale* stale;
  const float* rs_f;
  const double* rs_d;
  double alpha;
  double* part;        // [block][C - 1] gain sums
  float* sel_v;        // [level][block][kTopK]
  int* sel_id;
  RunDev* d;
};

template <typename T>
__device__ __forceinline__ float f_up(T x) {
  if constexpr (sizeof(T) == 8) return __double2float_ru(x);
  else return x;
}
template <typename T>
__device__ __forceinline__ float f_down(T x) {
  if constexpr (sizeof(T) == 8) return __double2float_rd(x);
  else return x;
}
template <typename T>
__device__ __forceinline__ T pos(T x) {
  return x > T(0) ? x : T(0);
}

// Merges the block lists of one level on one warp: the kTopK best heads, then the entries of their
// blocks (any other block's head has kTopK better entries ahead of it).
__device__ __forceinline__ void merge_level(const float* __restrict__ sel_v, const int* __restrict__ sel_id, int blocks,
                                            LevelSel* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  constexpr int NH = (kMeetBlocks + 31) / 32;
  float hv[NH];  // all the loads first: one round trip
  int hi[NH];
#pragma unroll
  for (int k = 0; k < NH; ++k) {
    const int blk = k * 32 + lane;
    const bool ok = blk < blocks;
    hv[k] = ok ? __ldcg(sel_v + static_cast<size_t>(blk) * kTopK) : -1.0f;
    hi[k] = ok ? __ldcg(sel_id + static_cast<size_t>(blk) * kTopK) : INT_MAX;
  }
  WarpList h;
#pragma unroll
  for (int k = 0; k < NH; ++k)
    if (k * 32 < blocks) warp_list_offer(h, hi[k] != INT_MAX, hv[k], hi[k], k * 32 + lane);
  constexpr int NE = kTopK / 2;
  float ev[NE];
  int ei[NE];
#pragma unroll
  for (int k = 0; k < NE; ++k) {
    const int src = 2 * k + (lane >> 4);
    const int tag = __shfl_sync(kFullMask, h.tag, src);
    const bool ok = __shfl_sync(kFullMask, h.id, src) != INT_MAX;
    const size_t e = static_cast<size_t>(ok ? tag : 0) * kTopK + (lane & 15);
    ev[k] = ok ? __ldcg(sel_v + e) : -1.0f;
    ei[k] = ok ? __ldcg(sel_id + e) : INT_MAX;
  }
  WarpList f;
#pragma unroll
  for (int k = 0; k < NE; ++k) warp_list_offer(f, ei[k] != INT_MAX, ev[k], ei[k], 0);
  if (lane < kTopK) {
    out->val[lane] = f.v;
    out->id[lane] = f.id;
  }
}

// A block's lists (one per warp and level) to sel_v / sel_id: warp l merges level l.
template <int NL>
__device__ __forceinline__ void block_levels(WarpList (&w)[NL], float* sv, int* si, float* __restrict__ sel_v,
                                             int* __restrict__ sel_id) {
  constexpr int NW = kThreads / 32;
  static_assert(NL <= NW, "one warp per level");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int l = 0; l < NL; ++l)
    if (lane < kTopK) {
      sv[(l * NW + warp) * kTopK + lane] = w[l].v;
      si[(l * NW + warp) * kTopK + lane] = w[l].id;
    }
  __syncthreads();
  if (warp < NL) {
    WarpList f;
#pragma unroll
    for (int j = 0; j < NW; j += 2) {
      const int e = (warp * NW + j + (lane >> 4)) * kTopK + (lane & 15);
      warp_list_offer(f, si[e] != INT_MAX, sv[e], si[e], 0);
    }
    if (lane < kTopK) {
      const size_t o = (static_cast<size_t>(warp) * gridDim.x + blockIdx.x) * kTopK + lane;
      sel_v[o] = f.v;
      sel_id[o] = f.id;
    }
  }
}

// The meeting pass: one thread per row adds up the row's stored vectors x_1..x_H (coalesced, each
// read once) and forms the candidates' gain terms and, with SEL, every level's bound; the best
// kTopK unevaluated vertices of each level go to out->lv. In a chain level d stands under
// T_d = S + {c_1..c_d}, phi(T_d) = column 0 - columns 1..d (a walk that avoids S avoids c_1..c_d or
// has a first c_j among them, counted in column j); differences are clamped at 0, and a vertex
// without a neighbour outside T_d (an exact count) has bound exactly 0. The last block to finish
// merges the lists and adds the gain sums in block order.
//
// Meant to stream H rows of the vectors (R-MAT scale 22: 384 MB, 57 us at the copy rate). Bounds and
// offers for seven levels cost five times that, so a warp skips them where none of its 32 rows can
// enter any level's list: bounds fall with the level, so the first level's bound without its
// correction, against the lowest last entry of the lists, decides. The rows come by decreasing
// degree, so after a warp's first iteration few pass. A bound of exactly 0 matters only when every
// bound is 0, so its vertex is recorded only while the warp's list is empty, and by one atomic per block
// (one per row, all to one address, serialise: k = 1 on a star of 100,000 leaves, 0.44 ms). R-MAT scale 22:
// 279 -> 123 us with FP32 gain terms, 180 us with pairs (97 M warp instructions instead of 42 M bound it, at 37% of
// the warps: a row's vectors, their low parts and the sums take the registers; 417 MB of traffic). On 10^5
// rows, where a warp has one iteration, the lists cost most (device_util.cuh): 97 -> 77 us.
template <typename T, int C, bool CHAIN, bool SEL, bool DIR>
__global__ void __launch_bounds__(kThreads, DIR || sizeof(T) * C > 32 ? 2 : kMeetPerSM) meet_kernel(const MeetArgs a) {
  constexpr int D = C - 1;
  constexpr int NL = CHAIN ? D : 1;
  constexpr int NW = kThreads / 32;
  __shared__ int s_cand[D];
  __shared__ float sv[SEL ? NL * NW * kTopK : 1];
  __shared__ int si[SEL ? NL * NW * kTopK : 1];
  __shared__ double sg[NW][D];
  __shared__ unsigned long long s_zero[SEL ? NL : 1];  // the block's smallest vertex with bound 0, per level
  __shared__ int is_last;
  const RunIn& in = a.d->in;
  if (SEL && threadIdx.x < NL) s_zero[threadIdx.x] = kNoZero;
  if (threadIdx.x < D) s_cand[threadIdx.x] = in.cand[threadIdx.x];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int H = a.H;
  const bool odd = (a.L & 1) != 0;
  const T* __restrict__ xs = static_cast<const T*>(a.xs);
  const T* __restrict__ rs = sizeof(T) == 8 ? reinterpret_cast<const T*>(a.rs_d) : reinterpret_cast<const T*>(a.rs_f);
  // directed rounding keeps a bound above that of the stored vectors; e covers the vectors' own
  // rounding where differences of columns cancel (sweeps' errors are independent and average over a row's
  // neighbours, so like the root of their number), keep the returns' where they reduce f
  const float e = sweep_rounding<T>() * sqrtf(fmaxf(1.0f, 0.25f * static_cast<float>(H - 1)));
  constexpr float keep = 1.0f - 2e-6f;
  const float infl = __fadd_ru(1.0f, __fmul_ru(static_cast<float>(H), 1.2e-7f));
  const float al2 = __double2float_rd(a.alpha * a.alpha), al3 = __double2float_ru(a.alpha * a.alpha * a.alpha);
  const int step = in.step;
  bool sampling = false;
  if (SEL) {
#pragma unroll
    for (int l = 0; l < NL; ++l) sampling |= in.thr[l] != ~0ull;
  }
  using W = WideOf<T>;
  Wide<T> acc[D] = {};
  WarpList w[NL];
  int nsampled[NL];
#pragma unroll
  for (int l = 0; l < NL; ++l) nsampled[l] = 0;
  float enter = -1.0f;     // lowest last entry of the warp's lists (-1: one is not full)
  unsigned empty = ~0u;    // levels whose list is empty
  const int32_t stride = gridDim.x * kThreads;
  for (int32_t base = blockIdx.x * kThreads + warp * 32; base < a.n_scan; base += stride) {
    const int32_t v = base + lane;
    const bool ok = v < a.n_scan;
    const bool has = v < a.n_active;
    const T* __restrict__ row = xs + static_cast<size_t>(has ? v : 0) * C;
    // the row's sums over t = 1..H-1 with their low parts, and x_H (directed: Br, xr of the walks that end here)
    T B[C], Bl[C], xh[C], Br[DIR ? C : 1], Brl[DIR ? C : 1], xr[DIR ? C : 1];
#pragma unroll
    for (int c = 0; c < C; ++c) B[c] = Bl[c] = xh[c] = T(0);
    if constexpr (DIR) {
#pragma unroll
      for (int c = 0; c < C; ++c) Br[c] = Brl[c] = xr[c] = T(0);
    }
    T inv = T(1);
    Wide<T> winv = W::make(T(1), T(0));
    if (has) {
      auto load = [&](const T* p, T (&x)[C]) {
        if constexpr (sizeof(T) * C >= 16) {
#pragma unroll
          for (int k = 0; k < static_cast<int>(sizeof(T)) * C / 16; ++k) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(p) + k);
            memcpy(&x[k * (16 / static_cast<int>(sizeof(T)))], &q, 16);
          }
        } else {
#pragma unroll
          for (int c = 0; c < C; ++c) x[c] = __ldg(p + c);
        }
      };
      const T* p = row;
#pragma unroll 4
      for (int t = 1; t < H; ++t, p += a.stride) {
        T x[C];
        load(p, x);
#pragma unroll
        for (int c = 0; c < C; ++c) W::accumulate(B[c], Bl[c], x[c]);
      }
      load(p, xh);
      if constexpr (DIR) {
        p = static_cast<const T*>(a.xr) + static_cast<size_t>(v) * C;
#pragma unroll 4
        for (int t = 1; t < H; ++t, p += a.stride) {
          T x[C];
          load(p, x);
#pragma unroll
          for (int c = 0; c < C; ++c) W::accumulate(Br[c], Brl[c], x[c]);
        }
        load(p, xr);
      }
      if (rs) {
        winv = W::inverse(rs[v]);
        inv = T(1) / rs[v];
      }
    }
    // gain terms of candidate d + 1 under its base set; nothing beyond the stored vectors is rounded to T
    {
      auto value = [&](T hi, T lo) { return rs ? W::make(hi, lo).times(winv) : W::make(hi, lo); };
      Wide<T> rb = value(B[0], Bl[0]), rh = value(xh[0], T(0)), sb = W::make(T(0), T(0)), sh = sb;
      if constexpr (DIR) {
        sb = W::make(Br[0], Brl[0]);
        sh = W::make(xr[0], T(0));
      }
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const Wide<T> kb = value(B[d + 1], Bl[d + 1]), kh = value(xh[d + 1], T(0));
        Wide<T> k = kb, vv, pp;
        k.add(kh);
        if constexpr (DIR) {
          const Wide<T> jh = W::make(xr[d + 1], T(0));
          vv = W::make(Br[d + 1], Brl[d + 1]);
          pp = sb;
          if (!odd) {
            vv.add(jh);
            pp.add(sh);
          }
          if (CHAIN) {
            sb.sub(W::make(Br[d + 1], Brl[d + 1]));
            sh.sub(jh);
          }
        } else {
          vv = odd ? kb : k;
          pp = rb;
          if (!odd) pp.add(rh);
        }
        pp = pp.pos();
        pp.sub(vv);
        acc[d].add(k);
        acc[d].add(vv.times(rh.pos()));
        acc[d].add(pp.pos().times(kh));
        if (CHAIN) {
          rb.sub(kb);
          rh.sub(kh);
        }
      }
    }
    if (rs) {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        B[c] *= inv;
        xh[c] *= inv;
      }
    }
    if (SEL) {
      bool out = false;
      int dg = 0, dr = 0;  // entries of the vertex's rows outside the level's set
      float tail = 0.0f;
      if (ok) {
        out = in_set(a.mask, v);
        if (has) {
          dg = a.g.rp[0][v + 1] - a.g.rp[0][v] - a.g.cnt[0][v];
          if (DIR) dr = a.g.rp[1][v + 1] - a.g.rp[1][v] - a.g.cnt[1][v];
          tail = a.tail[v];
        }
      }
      const float K0 = f_up(B[0] + xh[0]);
      const float most_u = __fmul_ru(K0, __fadd_ru(infl, e));
      float R0 = K0, most_f = most_u;
      if constexpr (DIR) {
        R0 = f_up(Br[0] + xr[0]);
        most_f = __fmul_ru(R0, __fadd_ru(infl, e));
      }
      const float most = dg + dr > 0 ? __fadd_ru(__fmaf_ru(most_f, most_u, __fadd_ru(most_f, most_u)), tail) : 0.0f;
      // some row of the warp may enter a list
      if (__any_sync(kFullMask, ok && !out && !(__fmul_ru(most, 1.00001f) < enter)) || a.bound) {
        bool evaluated = false;
        Stale st{0.0f, -1};
        uint32_t caller = 0;
        if (ok) {
          st = a.stale[v];
          if (sampling) caller = static_cast<uint32_t>(__ldg(a.perm + v));
          if (!CHAIN) {
#pragma unroll
            for (int j = 0; j < D; ++j) evaluated |= s_cand[j] == v;
          }
        }
        // a column's sums over t to H-1, H-2 and H-4, x_1, x_2 and x_H (what is not at hand read again
        // from the row: few warps come here on a large graph)
        struct Col {
          T b, b2, b4, f1, f2, h;
        };
        auto at = [&](int t, int c) {
          return has && t >= 1 ? __ldg(row + static_cast<size_t>(t - 1) * a.stride + c) * inv : T(0);
        };
        auto column = [&](int c) {
          Col k;
          k.f1 = at(1, c);
          k.f2 = H >= 2 ? at(2, c) : T(0);
          const T x1 = at(H - 1, c), x2 = at(H - 2, c), x3 = at(H - 3, c);
          k.b = B[c];
          k.h = xh[c];
          k.b2 = k.b - x1;
          k.b4 = k.b2 - x2 - x3;
          return k;
        };
        T eb = T(0), eh = T(0);  // directed: the level's walks that end here, to H-1 and of length H
        if constexpr (DIR) {
          eb = Br[0];
          eh = xr[0];
        }
        Col r = column(0);  // the level's phi
        const Col r0 = r;
#pragma unroll
        for (int d = 0; d < NL; ++d) {
          float ub = 0.0f;
          if (dg + dr > 0) {
            const float U = __fmaf_ru(f_up(pos(r.b + r.h)), infl, __fmul_ru(e, K0));
            float F, corr = 0.0f;
            if constexpr (DIR) {
              F = __fmaf_ru(f_up(pos(eb + eh)), infl, __fmul_ru(e, R0));
            } else {
              const float p1lo = fmaxf(0.0f, __fsub_rd(f_down(pos(r.f1)), e * f_up(r0.f1)));
              float s2, s4 = 0.0f;
              if (rs) {  // Cauchy-Schwarz: sum of squared weights >= (their sum)^2 / their number
                s2 = __fdiv_rd(__fmul_rd(p1lo, p1lo), static_cast<float>(dg));
              } else {
                s2 = __fmul_rd(al2, static_cast<float>(dg));
                const float p2lo = fmaxf(0.0f, __fsub_rd(f_down(pos(r.f2)), e * f_up(r0.f2)));
                const float p1up = __fadd_ru(f_up(pos(r.f1)), e * f_up(r0.f1));
                s4 = fmaxf(0.0f, __fsub_rd(__fmul_rd(al2, p2lo), __fmul_ru(al3, p1up)));
              }
              if (H >= 2) corr = __fmul_rd(s2, __fadd_rd(1.0f, fmaxf(0.0f, __fsub_rd(f_down(pos(r.b2)), e * f_up(r0.b2)))));
              if (H >= 4)
                corr = __fadd_rd(corr, __fmul_rd(s4, __fadd_rd(1.0f, fmaxf(0.0f, __fsub_rd(f_down(pos(r.b4)), e * f_up(r0.b4))))));
              corr = __fmul_rd(corr, keep);
              F = fmaxf(0.0f, __fsub_ru(U, corr));
            }
            ub = __fadd_ru(__fmaf_ru(F, U, __fadd_ru(F, U)), tail);
            if (odd) {  // the pair (H, H) is longer than L
              const float hlo = fmaxf(0.0f, __fsub_rd(f_down(pos(r.h)), e * f_up(r0.h)));
              float elo = hlo;
              if constexpr (DIR) elo = fmaxf(0.0f, __fsub_rd(f_down(pos(eh)), e * f_up(xr[0])));
              ub = __fsub_ru(ub, __fmul_rd(hlo, fmaxf(0.0f, __fsub_rd(elo, corr))));
            }
            if (!(ub >= 0.0f)) ub = INFINITY;  // overflow: nothing is known
            if (st.step >= 0 && st.ub < ub) ub = st.ub;
          }
          if (d == NL - 1 && ok && a.bound) a.bound[v] = ub;
          bool want = ok && !out;
          if (want && in.thr[d] != ~0ull) want = sample_hash(in.seed, static_cast<uint32_t>(step + d), caller) < in.thr[d];
          nsampled[d] += want;
          want = want && st.step != step + d && !(CHAIN ? s_cand[d] == v : evaluated);
          if (want && ub == 0.0f && (empty >> d & 1u)) {
            const unsigned long long z =
                (static_cast<unsigned long long>(__ldg(a.perm + v)) << 32) | static_cast<uint32_t>(v);
            if (z < s_zero[d]) atomicMin(&s_zero[d], z);
          }
          warp_list_offer(w[d], want && ub != 0.0f, ub, v, 0);
          if ((empty >> d & 1u) && __shfl_sync(kFullMask, w[d].id, 0) != INT_MAX) empty &= ~(1u << d);
          if (CHAIN && d + 1 < NL) {
            const Col k = column(d + 1);
            r.b -= k.b;
            r.b2 -= k.b2;
            r.b4 -= k.b4;
            r.f1 -= k.f1;
            r.f2 -= k.f2;
            r.h -= k.h;
            dg -= k.f1 > T(0);
            if constexpr (DIR) {
              eb -= Br[d + 1];
              eh -= xr[d + 1];
              dr -= has && __ldg(static_cast<const T*>(a.xr) + static_cast<size_t>(v) * C + d + 1) > T(0);
            }
            out |= s_cand[d] == v;
          }
        }
        enter = INFINITY;
#pragma unroll
        for (int l = 0; l < NL; ++l) enter = fminf(enter, __shfl_sync(kFullMask, w[l].v, kTopK - 1));
      }
    }
  }
  // gain sums of the block
#pragma unroll
  for (int d = 0; d < D; ++d) {
    double x = acc[d].get();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFullMask, x, o);
    if (lane == 0) sg[warp][d] = x;
  }
  if (SEL) {
    if (sampling) {
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        int x = nsampled[l];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFullMask, x, o);
        if (lane == 0 && x) atomicAdd(&a.d->out.lv[l].sampled, x);
      }
    }
    block_levels<NL>(w, sv, si, a.sel_v, a.sel_id);
  }
  __syncthreads();
  if (SEL && threadIdx.x < NL && s_zero[threadIdx.x] != kNoZero)
    atomicMin(&a.d->out.lv[threadIdx.x].zero_min, s_zero[threadIdx.x]);
  if (threadIdx.x < D) {
    double x = 0.0;
    for (int i = 0; i < NW; ++i) x += sg[i][threadIdx.x];
    a.part[static_cast<size_t>(blockIdx.x) * D + threadIdx.x] = x;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(&a.d->done, 1) == static_cast<int>(gridDim.x) - 1;
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  const int blocks = static_cast<int>(gridDim.x);
  if (SEL) {
    if (warp < NL)
      merge_level(a.sel_v + static_cast<size_t>(warp) * blocks * kTopK, a.sel_id + static_cast<size_t>(warp) * blocks * kTopK,
                  blocks, &a.d->out.lv[warp]);
  }
  for (int d = warp; d < D; d += NW) {
    double x = 0.0;
    for (int b = lane; b < blocks; b += 32) x += __ldcg(a.part + static_cast<size_t>(b) * D + d);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFullMask, x, o);
    if (lane == 0) {
      a.d->out.gains[d] = x;
      // exact under S (a chain's deeper levels stand under larger sets: no bound yet)
      if (SEL && s_cand[d] >= 0 && (!CHAIN || d == 0)) a.stale[s_cand[d]] = Stale{__double2float_ru(x), step};
    }
  }
}

// Selections of kRunLevels steps' samples (or, without sampling, one of all) from stored bounds: a
// choice of guesses, so the bounds may belong to an earlier set.
__global__ void __launch_bounds__(kThreads) guess_kernel(const float* __restrict__ bound, int32_t n_scan, int32_t n_active,
                                                         const uint32_t* __restrict__ mask,
                                                         const int32_t* __restrict__ perm, int levels,
                                                         float* __restrict__ sel_v, int* __restrict__ sel_id,
                                                         RunDev* __restrict__ d) {
  constexpr int NW = kThreads / 32;
  __shared__ float sv[kRunLevels * NW * kTopK];
  __shared__ int si[kRunLevels * NW * kTopK];
  __shared__ int is_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  WarpList w[kRunLevels];
  const int32_t stride = gridDim.x * kThreads;
  for (int32_t base = blockIdx.x * kThreads + warp * 32; base < n_scan; base += stride) {
    const int32_t v = base + lane;
    const bool live = v < n_scan && v < n_active && !in_set(mask, v);
    const float b = live ? bound[v] : 0.0f;
    const uint32_t caller = live ? static_cast<uint32_t>(__ldg(perm + v)) : 0u;
#pragma unroll
    for (int l = 0; l < kRunLevels; ++l) {
      if (l >= levels) break;
      bool want = live && b > 0.0f;
      if (want && d->in.thr[l] != ~0ull)
        want = sample_hash(d->in.seed, static_cast<uint32_t>(d->in.step + l), caller) < d->in.thr[l];
      warp_list_offer(w[l], want, b, v, 0);
    }
  }
  block_levels<kRunLevels>(w, sv, si, sel_v, sel_id);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(&d->done, 1) == static_cast<int>(gridDim.x) - 1;
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  const int blocks = static_cast<int>(gridDim.x);
  if (warp < kRunLevels)
    merge_level(sel_v + static_cast<size_t>(warp) * blocks * kTopK, sel_id + static_cast<size_t>(warp) * blocks * kTopK, blocks,
                &d->out.lv[warp]);
}

// Scoring run, first stored vector, rows [0, n_active): (h, m) pairs. Unweighted: x_1 from the
// counts: h_1 = alpha |N(v) cap S| (all of alpha deg on S), m_1 = alpha |N(v) \ S| (0 on S). Weighted
// (rs): x_0 = the indicators of S and V \ S, scaled.
template <typename T>
__global__ void pair_init(T* __restrict__ X, const int32_t* __restrict__ rp, const int32_t* __restrict__ cnt,
                          const uint32_t* __restrict__ mask, int32_t n_active, T alpha, const T* __restrict__ rs,
                          int32_t* __restrict__ done) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *done = 0;
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n_active; v += gridDim.x * blockDim.x) {
    const bool inS = in_set(mask, v);
    T h, m;
    if (rs) {
      h = inS ? rs[v] : T(0);
      m = inS ? T(0) : rs[v];
    } else {
      const int32_t dg = rp[v + 1] - rp[v], c = cnt[v];
      h = alpha * static_cast<T>(inS ? dg : c);
      m = inS ? T(0) : alpha * static_cast<T>(dg - c);
    }
    if constexpr (sizeof(T) == 4) reinterpret_cast<float2*>(X)[v] = make_float2(h, m);
    else reinterpret_cast<double2*>(X)[v] = make_double2(h, m);
  }
}

// Walks of length a + b that hit S: the half of length a hits, or it misses and the half of length b
// hits, so with b = H the lengths H + a, a = 1..L-H, number sum_v [h_a (h_H + m_H) + m_a h_H] and the
// lengths up to H are plain sums of h_t. One thread per row; the last block adds the block sums.
// x_t sits at slot (t - 1) % ring; with folded > 0 the two slots behind the ring hold x_1 + .. + x_folded (hi
// and lo parts). Nothing beyond the stored vectors is rounded to FP32.
template <typename T>
__global__ void __launch_bounds__(kThreads) pair_meet(const T* __restrict__ xs, int64_t stride, int32_t ring, int32_t folded,
                                                      int32_t L, int32_t H, int32_t n_active, const T* __restrict__ rs,
                                                      double* __restrict__ part, int32_t* __restrict__ done,
                                                      double* __restrict__ out) {
  constexpr int NW = kThreads / 32;
  __shared__ double sg[NW];
  __shared__ int is_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool odd = (L & 1) != 0;
  using W = WideOf<T>;
  Wide<T> acc = W::make(T(0), T(0));
  for (int32_t v = blockIdx.x * kThreads + threadIdx.x; v < n_active; v += gridDim.x * kThreads) {
    T bh = T(0), bm = T(0), lh = T(0), lm = T(0), h = T(0), m = T(0);  // sums over t < H and their low parts
    const T* row = xs + 2 * static_cast<size_t>(v);
    if (folded > 0) {
      const T* f = row + stride * ring;
      bh = f[0];
      bm = f[1];
      lh = f[stride];
      lm = f[stride + 1];
    }
#pragma unroll 4
    for (int t = folded + 1; t <= H; ++t) {
      const T* p = row + stride * ((t - 1) % ring);
      T xh, xm;
      if constexpr (sizeof(T) == 4) {
        const float2 q = __ldcs(reinterpret_cast<const float2*>(p));
        xh = q.x;
        xm = q.y;
      } else {
        const double2 q = __ldcs(reinterpret_cast<const double2*>(p));
        xh = q.x;
        xm = q.y;
      }
      if (t < H) {
        W::accumulate(bh, lh, xh);
        W::accumulate(bm, lm, xm);
      } else {
        h = xh;
        m = xm;
      }
    }
    Wide<T> vh = W::make(bh, lh), vm = W::make(bm, lm), wh = W::make(h, T(0)), wm = W::make(m, T(0));
    if (rs) {
      const Wide<T> inv = W::inverse(rs[v]);
      vh = vh.times(inv);
      vm = vm.times(inv);
      wh = wh.times(inv);
      wm = wm.times(inv);
    }
    Wide<T> k = vh, both = wh;
    k.add(wh);
    both.add(wm);
    if (!odd) {
      vh = k;
      vm.add(wm);
    }
    acc.add(k);
    acc.add(vh.times(both));
    acc.add(vm.times(wh));
  }
  double x = acc.get();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFullMask, x, o);
  if (lane == 0) sg[warp] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    x = 0.0;
    for (int i = 0; i < NW; ++i) x += sg[i];
    part[blockIdx.x] = x;
    __threadfence();
    is_last = atomicAdd(done, 1) == static_cast<int>(gridDim.x) - 1;
  }
  __syncthreads();
  if (!is_last || warp != 0) return;
  __threadfence();
  x = 0.0;
  for (int b = lane; b < static_cast<int>(gridDim.x); b += 32) x += __ldcg(part + b);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFullMask, x, o);
  if (lane == 0) *out = x;
}

// The sum behind the ring, hi and lo parts `stride` apart, (+)= x_{from+1} .. x_{from+count}, elementwise.
template <typename T>
__global__ void pair_fold(T* __restrict__ xs, int64_t stride, int32_t ring, int32_t from, int32_t count) {
  T* sum = xs + stride * ring;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < stride;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    T a = from > 0 ? sum[i] : T(0), lo = from > 0 ? sum[stride + i] : T(0);
    for (int32_t t = 0; t < count; ++t) WideOf<T>::accumulate(a, lo, xs[stride * ((from + t) % ring) + i]);
    sum[i] = a;
    sum[stride + i] = lo;
  }
}

int grid_of(int64_t n) { return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16))); }
// Blocks of join_kernel for a group of `count`, a power of two: few captured shapes.
dim3 join_grid(int64_t count, int32_t longest) {
  int x = 1;
  while (x * 8 < count && x < 2048) x *= 2;
  return dim3(x, longest > kJoinRow ? kChunks : 1);
}
int meet_grid(int32_t n_scan) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(kMeetBlocks, (int64_t(n_scan) + kThreads - 1) / kThreads)));
}

// The longest row of a graph, in either orientation.
int32_t longest_row(const Graph& g) { return std::max(g.dmax, g.rdmax); }

Rows rows_of(const Graph& g, const Workspace& ws) {
  Rows r{};
  r.rp[0] = g.rp.as<int32_t>();
  r.ci[0] = g.ci.as<int32_t>();
  r.cnt[0] = ws.cnt.as<int32_t>();
  r.directed = g.directed ? 1 : 0;
  if (g.directed) {
    r.rp[1] = g.rp_r.as<int32_t>();
    r.ci[1] = g.ci_r.as<int32_t>();
    r.cnt[1] = r.cnt[0] + g.n;
  }
  return r;
}

// X: the first stored vector; directed: that of the other set lies `set` elements behind it.
template <typename T, int C>
cudaError_t launch_init(cudaStream_t s, T* X, int64_t set, RunDev* d, const Graph& g, const Workspace& ws, bool chain,
                        double alpha) {
  const T* rs = !g.weighted ? nullptr : sizeof(T) == 8 ? static_cast<const T*>(g.rs_d.p) : static_cast<const T*>(g.rs_f.p);
  const Rows rows = rows_of(g, ws);
  const uint32_t* mask = ws.mask.as<uint32_t>();
  const T al = static_cast<T>(alpha);
  const int write = g.weighted ? 0 : 1, sets = g.directed ? 2 : 1;
  for (int o = 0; o < sets; ++o)
    run_init<T, C><<<grid_of(static_cast<int64_t>(g.n_active) * C * sizeof(T) / 16), 256, 0, s>>>(
        X + set * o, d, rows.rp[o], rows.cnt[o], mask, g.n_active, al, rs);
  if (chain) {
    run_scatter<T, true><<<dim3(kChunks, C - 1, sets), 256, 0, s>>>(X, set, C, d, rows, mask, al, write);
    run_own<T, true><<<sets, 32, 0, s>>>(X, set, C, d, rows, al, write);
  } else {
    if (write) run_scatter<T, false><<<dim3(kChunks, C - 1, sets), 256, 0, s>>>(X, set, C, d, rows, mask, al, write);
    run_own<T, false><<<sets, 32, 0, s>>>(X, set, C, d, rows, al, write);
  }
  return cudaGetLastError();
}

template <typename T, int C, bool CHAIN, bool SEL>
cudaError_t launch_meet(cudaStream_t s, const MeetArgs& a) {
  if (a.g.directed) meet_kernel<T, C, CHAIN, SEL, true><<<meet_grid(a.n_scan), kThreads, 0, s>>>(a);
  else meet_kernel<T, C, CHAIN, SEL, false><<<meet_grid(a.n_scan), kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

int64_t run_bytes(const Graph& g, int32_t L_max, int cols, bool fp64, bool select) {
  const int64_t n = g.n, H = (L_max + 1) / 2, es = fp64 ? 8 : 4, sets = g.directed ? 2 : 1;
  const int64_t slices = std::max(std::max(g.plan.num_slices, g.directed ? g.plan_r.num_slices : 0), 1);
  const int64_t heavy = std::max(std::max(g.plan.num_heavy, g.directed ? g.plan_r.num_heavy : 0), 1);
  // x_1 .. x_H (x_0: weighted)
  int64_t b = std::max<int64_t>(static_cast<int64_t>(g.n_active) * (sets * H + (g.weighted ? 1 : 0)) * cols * es, 16);
  b += n * 4 * sets + (n + 31) / 32 * 4;                    // counts of S in the rows, S bitmask
  b += static_cast<int64_t>(kMeetBlocks) * (cols - 1) * 8;  // gain sums
  b += static_cast<int64_t>(sizeof(RunDev)) + 256;
  if (select) b += n * (4 + 4 + static_cast<int64_t>(sizeof(Stale))) + static_cast<int64_t>(kMeetBlocks) * kRunLevels * kTopK * 8;
  return b + slices * cols * es + heavy * 4;
}

// The captured sequences copy from and to this block: it must outlive them at one address (a pinned
// block freed and made again at the same address is another allocation to the driver). Blocks go back to
// a pool (at most kIoPool, the rest are freed): pinning one takes longer than a run on a small graph.
namespace {
constexpr size_t kIoPool = 64;
std::mutex g_io_mu;
std::vector<void*>& io_pool() {
  static std::vector<void*>* p = new std::vector<void*>();  // lives until exit
  return *p;
}
}  // namespace

static gedwalk_status ensure_run_io(Workspace& ws) {
  if (ws.run_io) return GEDWALK_OK;
  {
    std::lock_guard<std::mutex> lk(g_io_mu);
    if (!io_pool().empty()) {
      ws.run_io = io_pool().back();
      io_pool().pop_back();
      return GEDWALK_OK;
    }
  }
  if (cudaMallocHost(&ws.run_io, sizeof(RunOut) + sizeof(RunIn)) != cudaSuccess) {
    cudaGetLastError();
    ws.run_io = nullptr;
    return fail(GEDWALK_ERR_OOM, "pinned host allocation of %zu bytes failed", sizeof(RunOut) + sizeof(RunIn));
  }
  return GEDWALK_OK;
}

void release_run_io(void* p) {
  if (!p) return;
  {
    std::lock_guard<std::mutex> lk(g_io_mu);
    if (io_pool().size() < kIoPool) {
      io_pool().push_back(p);
      return;
    }
  }
  cudaFreeHost(p);
}

gedwalk_status RunEngine::setup(int32_t L_max, int cols, bool select, const std::vector<int32_t>& init) {
  const size_t n = static_cast<size_t>(g.n), H_max = static_cast<size_t>((L_max + 1) / 2), es = r.fp64 ? 8 : 4;
  const size_t row = static_cast<size_t>(g.n_active) * cols * es;
  const size_t sets = g.directed ? 2 : 1;
  GW_TRY(ws.xs.ensure(row * (sets * H_max + (g.weighted ? 1 : 0)), s));
  GW_TRY(ws.cnt.ensure(sets * n * sizeof(int32_t), s));
  const size_t words = (n + 31) / 32;
  GW_TRY(ws.mask.ensure(words * 4, s));
  GW_TRY(ws.parts.ensure(static_cast<size_t>(kMeetBlocks) * (cols - 1) * sizeof(double), s));
  GW_TRY(ws.small.ensure(sizeof(RunDev) + 256, s));
  GW_TRY(ensure_run_io(ws));
  out = static_cast<RunOut*>(ws.run_io);
  in = reinterpret_cast<RunIn*>(out + 1);
  memset(in, 0, sizeof *in);
  for (uint64_t& t : in->thr) t = ~0ull;
  const int32_t slices = std::max(g.plan.num_slices, g.directed ? g.plan_r.num_slices : 0);
  const int32_t heavy = std::max(g.plan.num_heavy, g.directed ? g.plan_r.num_heavy : 0);
  GW_TRY(ws.partial.ensure(static_cast<size_t>(std::max(slices, 1)) * cols * es, s));
  const size_t cbytes = static_cast<size_t>(std::max(heavy, 1)) * sizeof(unsigned);
  if (ws.counters.bytes < cbytes || !ws.counters.p) GW_TRY(ws.counters.ensure(cbytes, s, /*zero=*/true));
  if (select) {
    GW_TRY(ws.stale.ensure(n * sizeof(Stale), s));
    GW_TRY(ws.sel.ensure(static_cast<size_t>(kMeetBlocks) * kRunLevels * kTopK * 8, s));
    GW_TRY(ws.tail.ensure(n * sizeof(float), s));
    GW_TRY(ws.bound.ensure(n * sizeof(float), s));
    GW_CUDA(cudaMemsetAsync(ws.stale.p, 0xff, n * sizeof(Stale), s));  // step -1
  }
  GW_CUDA(cudaMemsetAsync(ws.cnt.p, 0, sets * n * sizeof(int32_t), s));
  GW_CUDA(cudaMemsetAsync(ws.mask.p, 0, words * 4, s));
  if (!init.empty()) {
    DevBuf& list = ws.members;
    GW_TRY(list.ensure(init.size() * sizeof(int32_t), s));
    GW_TRY(ws.ensure_pinned(init.size() * sizeof(int32_t)));
    int32_t* st = static_cast<int32_t*>(ws.pinned);
    std::copy(init.begin(), init.end(), st);
    GW_CUDA(cudaMemcpyAsync(list.p, st, init.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
    join_kernel<<<join_grid(init.size(), longest_row(g)), 256, 0, s>>>(list.as<int32_t>(), static_cast<int32_t>(init.size()),
                                                                      rows_of(g, ws), ws.mask.as<uint32_t>());
    GW_KCHECK();
  }
  return GEDWALK_OK;
}

gedwalk_status RunEngine::set_length(int32_t length, bool select) {
  L = length;
  H = (L + 1) / 2;
  if (!select || g.n_active == 0) return GEDWALK_OK;
  // tail bounds from the walk totals; the tables are read under their lock, to the end of the kernel
  const int32_t rows = walk_rows(g, L + 1);
  // the largest entries of rows 1..L-H (the selections' lists are free here)
  unsigned long long* M = ws.sel.as<unsigned long long>();
  auto tails = [&](const double* A, const double* B) -> gedwalk_status {
    const double* rs = g.weighted ? g.rs_d.as<double>() : nullptr;
    if (!g.directed) {
      GW_CUDA(cudaMemsetAsync(M, 0, sizeof(*M) * (L - H + 1), s));
      if (L > H) {
        row_max_kernel<<<dim3(std::min(grid_of(g.n_active), 304), L - H), 256, 0, s>>>(A, g.n, g.n_active, rs, M);
        GW_KCHECK();
      }
    }
    tail_kernel<double><<<grid_of(g.n_active), 256, 0, s>>>(A, B, g.directed ? nullptr : reinterpret_cast<const double*>(M),
                                                            g.n, g.n_active, L, H, rs, r.alpha, 1.0 + 1e-12,
                                                            ws.tail.as<float>(), ws.bound.as<float>());
    GW_KCHECK();
    return GEDWALK_OK;
  };
  bool table;
  {
    std::shared_lock<std::shared_mutex> rl(g.tt_lock);
    table = g.tt_alpha == r.alpha && g.tt_rows >= rows;
  }
  if (table && g.directed) GW_TRY(ensure_totals_fwd(g, ws, r.alpha, rows, s));
  {
    std::shared_lock<std::shared_mutex> rl(g.tt_lock);
    if (g.tt_alpha == r.alpha && g.tt_rows >= rows && (!g.directed || (g.ttf_alpha == r.alpha && g.ttf_rows >= rows))) {
      GW_TRY(tails(g.directed ? g.ttab_f.as<double>() : g.ttab.as<double>(), g.ttab.as<double>()));
      GW_CUDA(cudaStreamSynchronize(s));
      return GEDWALK_OK;
    }
  }
  return r.fp64 ? own_tails<double>() : own_tails<float>();
}

// No table for this alpha (a forced L beyond the bound's reach): totals of this call's own, of the walks that
// avoid the S it starts from, to the full length (where walks multiply with their length the largest
// entries of the other form are far off) and in the runs' precision: in FP64 R-MAT scale 20, L = 9, spent
// 1.2 ms on them, more than on the run.
template <typename T>
gedwalk_status RunEngine::own_tails() {
  const size_t cells = static_cast<size_t>(L + 1) * g.n;
  const int sets = g.directed ? 2 : 1;
  GW_TRY(ws.ztab.ensure(sets * cells * sizeof(T), s));
  GW_TRY(ws.x0.ensure(static_cast<size_t>(g.n) * sizeof(T), s));  // the sweeps' unscaled values, unused
  T* tab = ws.ztab.as<T>();
  const T* rs = !g.weighted ? nullptr : sizeof(T) == 8 ? static_cast<const T*>(g.rs_d.p) : static_cast<const T*>(g.rs_f.p);
  for (int o = 0; o < sets; ++o) {
    T* row = tab + o * cells;
    own_row0<T><<<grid_of(g.n_active), 256, 0, s>>>(row, ws.mask.as<uint32_t>(), g.n_active, rs);
    GW_KCHECK();
    SweepArgs a = o ? base_args_rev(g, ws) : base_args(g, ws);
    a.alpha = r.alpha;
    a.Mout = ws.x0.p;
    for (int32_t t = 1; t <= L; ++t, row += g.n) {
      a.X = row;
      a.Y = row + g.n;
      GW_TRY(launch_sweep(MODE_MISS, sizeof(T) == 8, 1, a, s));
    }
  }
  // a sweep rounds a value by at most 41 units (run.h), and two values meet
  const double grow = 1.0 + 2.0 * (L + 1) * (sizeof(T) == 8 ? 5e-15 : 2.5e-6);
  tail_kernel<T><<<grid_of(g.n_active), 256, 0, s>>>(tab, tab + (sets - 1) * cells, nullptr, g.n, g.n_active, L, H, rs, r.alpha,
                                                     grow, ws.tail.as<float>(), ws.bound.as<float>());
  GW_KCHECK();
  return GEDWALK_OK;
}

void RunEngine::stale(int32_t v, double gain, int32_t step) {
  if (in->n_stale == kRunCols) return;  // a bound the passes then do without
  in->stale_id[in->n_stale] = v;
  in->stale_gain[in->n_stale] = gain;
  in->stale_step[in->n_stale++] = step;
}

// More joined vertices than a run carries go ahead of it.
gedwalk_status RunEngine::push_added() {
  RunDev* d = ws.small.as<RunDev>();
  while (added.size() > kRunCols) {
    std::copy(added.end() - kRunCols, added.end(), in->added);
    GW_CUDA(cudaMemcpyAsync(d->in.added, in->added, sizeof in->added, cudaMemcpyHostToDevice, s));
    join_kernel<<<join_grid(kRunCols, longest_row(g)), 256, 0, s>>>(d->in.added, kRunCols, rows_of(g, ws),
                                                                   ws.mask.as<uint32_t>());
    GW_KCHECK();
    GW_CUDA(cudaStreamSynchronize(s));  // the pinned block is reused
    added.resize(added.size() - kRunCols);
  }
  in->n_added = static_cast<int32_t>(added.size());
  std::copy(added.begin(), added.end(), in->added);
  added.clear();
  return GEDWALK_OK;
}

gedwalk_status RunEngine::issue(bool chain, int cols, bool select, bool profile, const std::vector<cudaEvent_t>* ev) {
  RunDev* d = ws.small.as<RunDev>();
  const bool fp64 = r.fp64;
  const size_t es = fp64 ? 8 : 4;
  const size_t row = static_cast<size_t>(g.n_active) * cols;
  GW_CUDA(cudaMemcpyAsync(&d->in, in, sizeof(RunIn), cudaMemcpyHostToDevice, s));
  run_begin<<<dim3(kChunks, kRunCols), 256, 0, s>>>(d, rows_of(g, ws), ws.mask.as<uint32_t>(),
                                                    select ? ws.stale.as<Stale>() : nullptr);
  GW_KCHECK();
  // x_1 .. x_H; a weighted graph starts one sweep earlier, from x_0 behind them; a directed one has its
  // second set behind the first
  char* xs = ws.xs.as<char>();
  char* x0 = g.weighted ? xs + row * es * H : xs;
  const int64_t set = static_cast<int64_t>(row) * H;
#define GW_RUN(T, C) \
  if (fp64 == (sizeof(T) == 8) && cols == C) GW_CUDA((launch_init<T, C>(s, reinterpret_cast<T*>(x0), set, d, g, ws, chain, r.alpha)));
  GW_RUN(float, 2) GW_RUN(float, 4) GW_RUN(float, 8) GW_RUN(float, 16) GW_RUN(double, 2) GW_RUN(double, 4) GW_RUN(double, 8)
#undef GW_RUN
  for (int i = 0; i < (g.directed ? 4 : 3); ++i) count_launch();
  const int mode = chain ? MODE_LOOK : MODE_PAR;
  if (ev) GW_CUDA(cudaEventRecordWithFlags((*ev)[0], s, cudaEventRecordExternal));
  for (int o = 0; o < (g.directed ? 2 : 1); ++o) {
    SweepArgs a = o ? base_args_rev(g, ws) : base_args(g, ws);
    a.alpha = r.alpha;
    a.cand = d->in.cand;
    a.live = d->live[o];
    char* x = xs + static_cast<size_t>(set) * es * o;
    for (int32_t t = g.weighted ? 1 : 2; t <= H; ++t) {
      a.X = t == 1 ? x0 : x + row * es * (t - 2);
      a.Y = x + row * es * (t - 1);
      GW_TRY(launch_sweep(mode, fp64, cols, a, s, profile));
    }
  }
  if (ev) GW_CUDA(cudaEventRecordWithFlags((*ev)[1], s, cudaEventRecordExternal));
  MeetArgs m{};
  m.xs = xs;
  m.xr = xs + static_cast<size_t>(set) * es;
  m.stride = static_cast<int64_t>(row);
  m.L = L;
  m.H = H;
  m.n_scan = select ? n_scan : g.n_active;
  m.n_active = g.n_active;
  m.g = rows_of(g, ws);
  m.mask = ws.mask.as<uint32_t>();
  m.perm = g.perm_d.as<int32_t>();
  m.tail = ws.tail.as<float>();
  m.bound = draws ? ws.bound.as<float>() : nullptr;
  m.stale = ws.stale.as<Stale>();
  m.rs_f = g.weighted ? g.rs_f.as<float>() : nullptr;
  m.rs_d = g.weighted ? g.rs_d.as<double>() : nullptr;
  m.alpha = r.alpha;
  m.part = ws.parts.as<double>();
  m.sel_v = ws.sel.as<float>();
  m.sel_id = reinterpret_cast<int*>(m.sel_v + static_cast<size_t>(kMeetBlocks) * kRunLevels * kTopK);
  m.d = d;
#define GW_MEET(T, C, CH, SE) \
  if (fp64 == (sizeof(T) == 8) && cols == C && chain == CH && select == SE) GW_CUDA((launch_meet<T, C, CH, SE>(s, m)));
  GW_MEET(float, 4, true, true) GW_MEET(float, 8, true, true) GW_MEET(double, 4, true, true) GW_MEET(double, 8, true, true)
  GW_MEET(float, 2, false, true) GW_MEET(float, 4, false, true) GW_MEET(float, 8, false, true)
  GW_MEET(double, 2, false, true) GW_MEET(double, 4, false, true) GW_MEET(double, 8, false, true)
  GW_MEET(float, 2, false, false) GW_MEET(float, 4, false, false) GW_MEET(float, 8, false, false)
  GW_MEET(float, 16, false, false)
  GW_MEET(double, 2, false, false) GW_MEET(double, 4, false, false) GW_MEET(double, 8, false, false)
#undef GW_MEET
  count_launch();
  GW_CUDA(cudaMemcpyAsync(out, &d->out, sizeof(RunOut), cudaMemcpyDeviceToHost, s));
  return GEDWALK_OK;
}

gedwalk_status RunEngine::run(bool chain, int cols, bool select, const std::vector<int32_t>& cand) {
  for (int j = 0; j < kRunCols; ++j) in->cand[j] = j < static_cast<int>(cand.size()) && j < cols - 1 ? cand[j] : -1;
  GW_TRY(push_added());
  const int swept = g.weighted ? H : (g.directed ? 2 : 1) * (H - 1);
  sweeps += swept;
  const int mode = chain ? MODE_LOOK : MODE_PAR;
  uint64_t abits;
  memcpy(&abits, &r.alpha, 8);
  auto bits = [](const void* p) { return static_cast<uint64_t>(reinterpret_cast<uintptr_t>(p)); };
  Sequence q;
  q.key = mix_all({uint64_t(mode), uint64_t(cols), uint64_t(r.fp64), uint64_t(L), uint64_t(select), uint64_t(n_scan), uint64_t(draws), abits,
                   bits(&g), bits(s), bits(ws.xs.p), bits(ws.cnt.p), bits(ws.mask.p), bits(ws.parts.p), bits(ws.small.p),
                   bits(ws.partial.p), bits(ws.counters.p), bits(ws.stale.p), bits(ws.sel.p), bits(ws.tail.p),
                   bits(ws.bound.p), bits(ws.run_io), bits(g.rp.p), bits(g.ci.p), bits(g.plan.units.p)});
  q.kernels = (g.directed ? 6 : 5) + swept;
  q.sweeps = swept;
  q.bytes = sweep_bytes(mode, r.fp64, cols, g.n_active, g.nnz, g.weighted);
  q.prof_key = (mode * 1000 + cols) * 2 + (r.fp64 ? 1 : 0);
  q.nnz = g.nnz;
  GW_TRY(run_sequence(ws, s, q, [&](bool profile, const std::vector<cudaEvent_t>* ev) {
    return issue(chain, cols, select, profile, ev);
  }));
  GW_CUDA(cudaStreamSynchronize(s));
  read_graph_timing(ws);
  in->n_stale = 0;
  in->n_added = 0;
  return GEDWALK_OK;
}

gedwalk_status RunEngine::guess(int levels) {
  RunDev* d = ws.small.as<RunDev>();
  GW_TRY(push_added());
  GW_CUDA(cudaMemcpyAsync(&d->in, in, sizeof(RunIn), cudaMemcpyHostToDevice, s));
  run_begin<<<dim3(kChunks, kRunCols), 256, 0, s>>>(d, rows_of(g, ws), ws.mask.as<uint32_t>(), ws.stale.as<Stale>());
  GW_KCHECK();
  float* sel_v = ws.sel.as<float>();
  guess_kernel<<<meet_grid(n_scan), kThreads, 0, s>>>(
      ws.bound.as<float>(), n_scan, g.n_active, ws.mask.as<uint32_t>(), g.perm_d.as<int32_t>(), levels, sel_v,
      reinterpret_cast<int*>(sel_v + static_cast<size_t>(kMeetBlocks) * kRunLevels * kTopK), d);
  GW_KCHECK();
  GW_CUDA(cudaMemcpyAsync(out, &d->out, sizeof(RunOut), cudaMemcpyDeviceToHost, s));
  GW_CUDA(cudaStreamSynchronize(s));
  in->n_stale = 0;
  in->n_added = 0;
  return GEDWALK_OK;
}

gedwalk_status score_run(Graph& g, Workspace& ws, const std::vector<int32_t>& S_int, const Resolved& r_in, double* score) {
  Resolved r = r_in;
  GW_TRY(greedy_stream(ws, r_in.stream, &r.stream));
  struct Guard {  // nothing launched here still runs when a call leaves early
    cudaStream_t s;
    bool ok = false;
    ~Guard() {
      if (!ok) {
        cudaStreamSynchronize(s);
        cudaGetLastError();
      }
    }
  } guard{r.stream};
  cudaStream_t s = r.stream;
  const bool fp64 = r.fp64;
  const size_t n = static_cast<size_t>(g.n), es = fp64 ? 8 : 4;
  const int32_t H = (r.L + 1) / 2;
  const size_t row = static_cast<size_t>(g.n_active) * 2;
  GW_TRY(ensure_run_io(ws));
  // x_1 .. x_H, or, where they would outgrow kWideBytes or the device, a ring of the last ones (three at
  // least) and the sum of the older; x_0 (weighted) sits where x_ring goes later
  int32_t ring = static_cast<int32_t>(std::max<int64_t>(
      3, std::min<int64_t>(H + (g.weighted ? 1 : 0), kWideBytes / std::max<int64_t>(static_cast<int64_t>(row * es), 1))));
  for (;; ring = std::max(3, ring / 2)) {
    const gedwalk_status st = ws.xs.ensure(row * es * (ring + (H > ring ? 2 : 0)), s);
    if (st == GEDWALK_OK) break;
    if (st != GEDWALK_ERR_OOM || ring <= 3) return st;
  }
  GW_TRY(ws.cnt.ensure(n * sizeof(int32_t), s));
  const size_t words = (n + 31) / 32;
  GW_TRY(ws.mask.ensure(words * 4, s));
  GW_TRY(ws.parts.ensure(kMeetBlocks * sizeof(double), s));
  GW_TRY(ws.small.ensure(64, s));
  GW_TRY(ws.partial.ensure(static_cast<size_t>(std::max(g.plan.num_slices, 1)) * 2 * es, s));
  const size_t cbytes = static_cast<size_t>(std::max(g.plan.num_heavy, 1)) * sizeof(unsigned);
  if (ws.counters.bytes < cbytes || !ws.counters.p) GW_TRY(ws.counters.ensure(cbytes, s, /*zero=*/true));
  // the group: its size, then its members
  const int32_t count = static_cast<int32_t>(S_int.size());
  GW_TRY(ws.members.ensure((S_int.size() + 1) * sizeof(int32_t), s));
  GW_TRY(ws.ensure_pinned((S_int.size() + 1) * sizeof(int32_t)));
  int32_t* st = static_cast<int32_t*>(ws.pinned);
  st[0] = count;
  std::copy(S_int.begin(), S_int.end(), st + 1);
  GW_CUDA(cudaMemcpyAsync(ws.members.p, st, (S_int.size() + 1) * sizeof(int32_t), cudaMemcpyHostToDevice, s));
  const dim3 join = join_grid(count, longest_row(g));
  double* d_sum = ws.small.as<double>();
  int32_t* d_done = reinterpret_cast<int32_t*>(d_sum + 1);
  double* h_sum = static_cast<double*>(ws.run_io);
  auto issue = [&](bool profile, const std::vector<cudaEvent_t>* ev) -> gedwalk_status {
    GW_CUDA(cudaMemsetAsync(ws.cnt.p, 0, n * sizeof(int32_t), s));
    GW_CUDA(cudaMemsetAsync(ws.mask.p, 0, words * 4, s));
    join_kernel<<<join, 256, 0, s>>>(ws.members.as<int32_t>() + 1, -1, rows_of(g, ws), ws.mask.as<uint32_t>());
    GW_KCHECK();
    char* xs = ws.xs.as<char>();
    char* x0 = g.weighted ? xs + row * es * (ring - 1) : xs;
    if (fp64)
      pair_init<double><<<grid_of(g.n_active), 256, 0, s>>>(reinterpret_cast<double*>(x0), g.rp.as<int32_t>(),
                                                            ws.cnt.as<int32_t>(), ws.mask.as<uint32_t>(), g.n_active, r.alpha,
                                                            g.weighted ? g.rs_d.as<double>() : nullptr, d_done);
    else
      pair_init<float><<<grid_of(g.n_active), 256, 0, s>>>(reinterpret_cast<float*>(x0), g.rp.as<int32_t>(),
                                                           ws.cnt.as<int32_t>(), ws.mask.as<uint32_t>(), g.n_active,
                                                           static_cast<float>(r.alpha),
                                                           g.weighted ? g.rs_f.as<float>() : nullptr, d_done);
    GW_KCHECK();
    SweepArgs a = base_args(g, ws);
    a.alpha = r.alpha;
    if (ev) GW_CUDA(cudaEventRecordWithFlags((*ev)[0], s, cudaEventRecordExternal));
    int32_t folded = 0;
    for (int32_t t = g.weighted ? 1 : 2; t <= H; ++t) {
      if (t - folded > ring) {  // x_t takes the slot of x_{t-ring}: fold all before x_{t-1}
        const int32_t count = ring - 1;
        if (fp64)
          pair_fold<double><<<grid_of(static_cast<int64_t>(row)), 256, 0, s>>>(reinterpret_cast<double*>(xs),
                                                                              static_cast<int64_t>(row), ring, folded, count);
        else
          pair_fold<float><<<grid_of(static_cast<int64_t>(row)), 256, 0, s>>>(reinterpret_cast<float*>(xs),
                                                                             static_cast<int64_t>(row), ring, folded, count);
        GW_KCHECK();
        folded += count;
      }
      a.X = t == 1 ? x0 : xs + row * es * ((t - 2) % ring);
      a.Y = xs + row * es * ((t - 1) % ring);
      GW_TRY(launch_sweep(MODE_PAIR, fp64, 2, a, s, profile));
    }
    if (ev) GW_CUDA(cudaEventRecordWithFlags((*ev)[1], s, cudaEventRecordExternal));
    if (fp64)
      pair_meet<double><<<meet_grid(g.n_active), kThreads, 0, s>>>(reinterpret_cast<double*>(xs), static_cast<int64_t>(row), ring, folded, r.L,
                                                                   H, g.n_active,
                                                                   g.weighted ? g.rs_d.as<double>() : nullptr,
                                                                   ws.parts.as<double>(), d_done, d_sum);
    else
      pair_meet<float><<<meet_grid(g.n_active), kThreads, 0, s>>>(reinterpret_cast<float*>(xs), static_cast<int64_t>(row), ring, folded, r.L, H,
                                                                  g.n_active, g.weighted ? g.rs_f.as<float>() : nullptr,
                                                                  ws.parts.as<double>(), d_done, d_sum);
    GW_KCHECK();
    GW_CUDA(cudaMemcpyAsync(h_sum, d_sum, sizeof(double), cudaMemcpyDeviceToHost, s));
    return GEDWALK_OK;
  };
  const int swept = g.weighted ? H : H - 1;
  uint64_t abits;
  memcpy(&abits, &r.alpha, 8);
  auto bits = [](const void* p) { return static_cast<uint64_t>(reinterpret_cast<uintptr_t>(p)); };
  Sequence q;
  q.key = mix_all({uint64_t(MODE_PAIR), uint64_t(fp64), uint64_t(r.L), uint64_t(join.x), uint64_t(ring), abits, bits(&g), bits(s), bits(ws.xs.p),
                   bits(ws.cnt.p), bits(ws.mask.p), bits(ws.parts.p), bits(ws.small.p), bits(ws.partial.p),
                   bits(ws.counters.p), bits(ws.members.p), bits(ws.run_io), bits(g.rp.p), bits(g.ci.p), bits(g.plan.units.p)});
  q.kernels = 3 + swept + (H > ring ? (H - ring - 1) / (ring - 1) + 1 : 0);
  q.sweeps = swept;
  q.bytes = sweep_bytes(MODE_PAIR, fp64, 2, g.n_active, g.nnz, g.weighted);
  q.prof_key = (MODE_PAIR * 1000 + 2) * 2 + (fp64 ? 1 : 0);
  q.nnz = g.nnz;
  GW_TRY(run_sequence(ws, s, q, issue));
  GW_CUDA(cudaStreamSynchronize(s));
  read_graph_timing(ws);
  *score = *h_sum;
  guard.ok = true;
  return GEDWALK_OK;
}

}  // namespace gw
