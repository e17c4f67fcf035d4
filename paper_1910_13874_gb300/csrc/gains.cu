// Exact marginal gains of every vertex on a graph whose walk vectors fit one SM's shared memory.
//
// The gain of c needs the half-length column of walks through c (run.cu). All n columns share one
// small graph, so a block keeps its columns in shared memory from the first step to the last and no
// step waits for another block: one launch instead of n / 15 runs of ceil(L/2) sweeps each (Erdos-
// Renyi, n = 3001, degree 10, FP32: 23.2 ms, 5 us a sweep, nearly all of it launch and latency; now
// 1.32 ms). A block is bound by instructions and latency: an index load and a 4-byte shared load per lane
// and entry, five loads and some forty operations per row and step, one block of 32 warps per SM (the
// columns take 192 KB); the shared-memory gathers by themselves would take a quarter of the time.
#include <algorithm>

#include "run.h"

namespace gw {
namespace {

constexpr int kGainThreads = 1024;
constexpr int kGroup = 8;  // lanes of a short row (K columns, kGroup / K entries at a time)
constexpr int kParts = 8;  // partial sums a lane keeps of its entries of a row
constexpr size_t kGainSmem = 200 * 1024;

struct GainArgs {
  const int32_t* rp;
  const int32_t* ci;
  int32_t n_active, n_long;  // rows [0, n_long) take a warp each: above 64 entries, 32 with 8 columns
  int64_t phi_stride;
  const uint32_t* mask;
  const void* phi;  // phi_0 .. phi_H under S, true values
  int32_t L, H;
  double alpha;
  const float* rs_f;
  const double* rs_d;
  double* out;  // by internal id
};

// One step for one row on W lanes: lane l holds column l % K and the entries l / K, + W / K, .. in kParts
// partial sums taken in turn, so a row has kParts W / K of them, added up as a tree: as few additions in
// a row as the sweeps' (one running sum over 64 equal entries can drift by 16 units in the last place).
// Nothing else is rounded to FP32: the gain terms are pairs.
template <typename T, int K, int W>
__device__ __forceinline__ void gain_row(const GainArgs& a, const T* __restrict__ x, T* __restrict__ y,
                                         const T* __restrict__ phi1, const T* __restrict__ phi0,
                                         const T* __restrict__ rs, int32_t v, bool ok, int32_t c, int l, bool both,
                                         Wide<T>& acc) {
  const int col = l % K;
  T part[kParts];
#pragma unroll
  for (int p = 0; p < kParts; ++p) part[p] = T(0);
  if (ok) {
    const int64_t e1 = a.rp[v + 1];
    for (int64_t e = a.rp[v] + l / K; e < e1; e += kParts * (W / K)) {
#pragma unroll
      for (int p = 0; p < kParts; ++p)
        if (e + p * (W / K) < e1) part[p] += x[static_cast<size_t>(__ldg(a.ci + e + p * (W / K))) * K + col];
    }
  }
#pragma unroll
  for (int p = kParts / 2; p > 0; p /= 2)
#pragma unroll
    for (int q = 0; q < p; ++q) part[q] += part[q + p];
  T s = part[0];
#pragma unroll
  for (int o = K; o < W; o <<= 1) s += __shfl_xor_sync(kFullMask, s, o);
  if (!ok || l >= K) return;
  const bool inS = (__ldg(a.mask + (v >> 5)) >> (v & 31)) & 1u;
  const T sv = rs ? rs[v] : T(1);
  const T f1 = phi1[v], f0 = phi0[v];
  T k1 = inS ? T(0) : static_cast<T>(a.alpha) * sv * s;
  if (v == c) k1 = f1;
  const size_t i = static_cast<size_t>(v) * K + col;
  using WT = WideOf<T>;
  Wide<T> k0 = WT::make(x[i], T(0));
  if (rs) k0 = k0.times(WT::inverse(sv));
  // walks of length 2t - 1 (halves t and t - 1) and 2t (halves t and t)
  Wide<T> w = WT::make(f0, T(0));
  w.sub(k0);
  w = w.pos();
  if (both) {
    Wide<T> m1 = WT::make(f1, T(0));
    m1.sub(WT::make(k1, T(0)));
    w.add(f1);
    w.add(m1.pos());
  }
  acc.add(w.times(k1));
  acc.add(k0.times(f1));
  y[i] = k1 * sv;
}

template <typename T, int K>
__global__ void __launch_bounds__(kGainThreads) gains_kernel(const GainArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  T* x = reinterpret_cast<T*>(smem);
  T* y = x + static_cast<size_t>(a.n_active) * K;
  __shared__ double sums[kGainThreads / 32][K];
  const T* rs = sizeof(T) == 8 ? reinterpret_cast<const T*>(a.rs_d) : reinterpret_cast<const T*>(a.rs_f);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t first = static_cast<int32_t>(blockIdx.x) * K;
  for (int32_t i = threadIdx.x; i < a.n_active * K; i += kGainThreads) x[i] = T(0);
  __syncthreads();
  auto live = [&](int32_t c) { return c < a.n_active && !((__ldg(a.mask + (c >> 5)) >> (c & 31)) & 1u); };
  if (threadIdx.x < K && live(first + static_cast<int32_t>(threadIdx.x))) {
    const int32_t c = first + static_cast<int32_t>(threadIdx.x);
    x[static_cast<size_t>(c) * K + threadIdx.x] = rs ? rs[c] : T(1);
  }
  __syncthreads();
  int32_t c = first + lane % K;  // this lane's candidate
  if (!live(c)) c = -1;
  Wide<T> acc = WideOf<T>::make(T(0), T(0));
  constexpr int NW = kGainThreads / 32, GW = 32 / kGroup;
  for (int32_t t = 1; t <= a.H; ++t) {
    const T* phi1 = static_cast<const T*>(a.phi) + a.phi_stride * t;
    const T* phi0 = phi1 - a.phi_stride;
    const bool both = 2 * t <= a.L;
    for (int32_t v = warp; v < a.n_long; v += NW) gain_row<T, K, 32>(a, x, y, phi1, phi0, rs, v, true, c, lane, both, acc);
    for (int32_t v0 = a.n_long + warp * GW; v0 < a.n_active; v0 += NW * GW) {
      const int32_t v = v0 + lane / kGroup;
      gain_row<T, K, kGroup>(a, x, y, phi1, phi0, rs, v, v < a.n_active, c, lane % kGroup, both, acc);
    }
    __syncthreads();
    T* z = x;
    x = y;
    y = z;
  }
  double g = acc.get();
#pragma unroll
  for (int o = K; o < 32; o <<= 1) g += __shfl_xor_sync(kFullMask, g, o);
  if (lane < K) sums[warp][lane] = g;
  __syncthreads();
  if (threadIdx.x < K && first + static_cast<int32_t>(threadIdx.x) < a.n_active) {
    double s = 0.0;
    for (int w = 0; w < NW; ++w) s += sums[w][threadIdx.x];
    a.out[first + threadIdx.x] = c >= 0 ? s : 0.0;
  }
}

// phi_0 = 1_{V\S} (true) and the first gathered vector (scaled)
template <typename T>
__global__ void phi_init(T* __restrict__ phi0, T* __restrict__ x, const uint32_t* __restrict__ mask, int32_t n,
                         const T* __restrict__ rs) {
  for (int32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    const T m = ((mask[v >> 5] >> (v & 31)) & 1u) ? T(0) : T(1);
    phi0[v] = m;
    x[v] = rs ? m * rs[v] : m;
  }
}

template <typename T, int K>
gedwalk_status launch_gains(const GainArgs& a, cudaStream_t s) {
  const size_t bytes = 2 * static_cast<size_t>(a.n_active) * K * sizeof(T);
  GW_CUDA(cudaFuncSetAttribute(gains_kernel<T, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kGainSmem)));
  gains_kernel<T, K><<<(a.n_active + K - 1) / K, kGainThreads, bytes, s>>>(a);
  GW_KCHECK();
  return GEDWALK_OK;
}

}  // namespace

// Columns of a block, 0: the vectors do not fit. Two columns at least: with one, a gather brings four
// bytes and the graph's runs (run.cu) of 15 columns are about as fast.
int small_gain_cols(const Graph& g, bool fp64) {
  if (g.directed || g.n_active < 1) return 0;
  for (int k = 8; k >= 2; k /= 2)
    if (2 * static_cast<size_t>(g.n_active) * k * (fp64 ? 8 : 4) <= kGainSmem) return k;
  return 0;
}

gedwalk_status small_gains(Graph& g, Workspace& ws, const Resolved& r, const std::vector<int32_t>& S, double* out) {
  const cudaStream_t s = r.stream;
  const bool fp64 = r.fp64;
  const size_t n = static_cast<size_t>(g.n), es = fp64 ? 8 : 4;
  const int32_t H = (r.L + 1) / 2;
  GW_TRY(upload_mask(g, ws, S, s));
  GW_TRY(ws.mtab.ensure(n * (H + 1) * es, s));
  GW_TRY(ws.x0.ensure(n * es, s));
  GW_TRY(ws.x1.ensure(n * es, s));
  GW_TRY(ensure_sweep_scratch(g, ws, 1, fp64, s));
  GW_TRY(ws.members.ensure(n * sizeof(double), s));
  GW_TRY(ws.ensure_pinned(n * sizeof(double)));
  const int blocks = static_cast<int>(std::min<size_t>((n + 255) / 256, 1024));
  if (fp64)
    phi_init<double><<<blocks, 256, 0, s>>>(ws.mtab.as<double>(), ws.x0.as<double>(), ws.mask.as<uint32_t>(), g.n,
                                            g.weighted ? g.rs_d.as<double>() : nullptr);
  else
    phi_init<float><<<blocks, 256, 0, s>>>(ws.mtab.as<float>(), ws.x0.as<float>(), ws.mask.as<uint32_t>(), g.n,
                                           g.weighted ? g.rs_f.as<float>() : nullptr);
  GW_KCHECK();
  SweepArgs a = base_args(g, ws);
  a.alpha = r.alpha;
  void* cur = ws.x0.p;
  void* nxt = ws.x1.p;
  for (int32_t t = 1; t <= H; ++t) {
    a.X = cur;
    a.Y = nxt;
    a.Mout = ws.mtab.as<char>() + static_cast<size_t>(t) * n * es;
    GW_TRY(launch_sweep(MODE_MISS, fp64, 1, a, s));
    std::swap(cur, nxt);
  }
  GainArgs q{};
  q.rp = g.rp.as<int32_t>();
  q.ci = g.ci.as<int32_t>();
  q.n_active = g.n_active;
  q.n_long = small_gain_cols(g, fp64) == 8 ? g.plan.num_mid : g.plan.num_long;
  q.phi_stride = static_cast<int64_t>(n);
  q.mask = ws.mask.as<uint32_t>();
  q.phi = ws.mtab.p;
  q.L = r.L;
  q.H = H;
  q.alpha = r.alpha;
  q.rs_f = g.weighted ? g.rs_f.as<float>() : nullptr;
  q.rs_d = g.weighted ? g.rs_d.as<double>() : nullptr;
  q.out = ws.members.as<double>();
  const int k = small_gain_cols(g, fp64);
  gedwalk_status st;
  if (fp64) st = k == 8 ? launch_gains<double, 8>(q, s) : k == 4 ? launch_gains<double, 4>(q, s) : launch_gains<double, 2>(q, s);
  else st = k == 8 ? launch_gains<float, 8>(q, s) : k == 4 ? launch_gains<float, 4>(q, s) : launch_gains<float, 2>(q, s);
  GW_TRY(st);
  const size_t got = static_cast<size_t>(g.n_active) * sizeof(double);
  GW_CUDA(cudaMemcpyAsync(ws.pinned, q.out, got, cudaMemcpyDeviceToHost, s));
  GW_CUDA(cudaStreamSynchronize(s));
  memcpy(out, ws.pinned, got);
  return GEDWALK_OK;
}

}  // namespace gw
