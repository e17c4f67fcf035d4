// Allocation-free variant of the two-state scoring sweep.
//
// Some callers cannot allocate device memory at all: code that runs after its
// framework has handed every byte of the GPU to its own pool, or embedded services
// that forbid allocation (and its latency or failure) once they are serving. For
// them gedwalk_score_step_noalloc runs one step of the two-state hit/miss
// recurrence on device buffers the caller already owns. The only scratch it needs,
// the per-block FP64 partial sums of the hit column, lives in the file-scope array
// below, which every GPU that loads this library holds until the process exits.
#include <cuda_runtime.h>

#include <mutex>

#include "internal.h"

namespace gw {
namespace {

constexpr int kNaWarps = kThreads / 32;
constexpr int kNaLanes = 8;                         // lanes of a row
constexpr int kNaGroups = 32 / kNaLanes;            // rows a warp works on side by side
constexpr int kNaRowStep = kNaWarps * kNaGroups;    // rows of a block's iteration: 32
constexpr int kNaHub = 256;                         // longer rows take a warp each, after the others
constexpr int kNaChunk = 2048;                      // still longer ones the block, so many entries at a time
constexpr int kNaMaxBlocks = 8192;                  // 8192 doubles = 64 KiB
constexpr int64_t kNaMaxRows = int64_t(2048) * kNaMaxBlocks;  // 16,777,216
constexpr int kNaMaxHubs = 2048;                    // rows of the largest block
constexpr int kNaMaxDevices = 64;

// One FP64 partial sum per block of the largest launch. Shared by every call on a device:
// each call overwrites every slot it reads, so nothing has to start at zero.
static __device__ __align__(256) double g_na_slots[kNaMaxBlocks];

std::mutex g_na_mu;
double* g_na_ptr[kNaMaxDevices] = {};  // device address of g_na_slots, per device

// Every row sum has one order, whoever computes it: 32 strided partial sums (entry j goes to partial
// j mod 32, each added up in order), then halving, partial i + partial i + 16, then + 8, + 4, + 2, + 1.
// A group of 8 lanes holds partials l, l + 8, l + 16, l + 24 on lane l.
struct Part {
  float h[4], m[4];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = m[q] = 0.0f;
  }
  __device__ __forceinline__ void add(int q, float2 v) {
    h[q] += v.x;
    m[q] += v.y;
  }
  __device__ __forceinline__ float2 total() const {
    float a = (h[0] + h[2]) + (h[1] + h[3]), b = (m[0] + m[2]) + (m[1] + m[3]);
#pragma unroll
    for (int o = kNaLanes / 2; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    return make_float2(a, b);
  }
};

__device__ __forceinline__ double na_store(const uint32_t* __restrict__ mask, float2* __restrict__ y, int64_t r,
                                           float alpha, float sh, float sm) {
  const bool inS = (__ldg(mask + (r >> 5)) >> (r & 31)) & 1u;
  const float h = alpha * (inS ? sh + sm : sh);
  const float m = inS ? 0.0f : alpha * sm;
  y[r] = make_float2(h, m);
  return static_cast<double>(h);
}

// One step of Section 3.1.1 on x = (hit, miss) pairs:
//   hit'(v)  = alpha (sum_{u~v} hit(u) + [v in S] sum_{u~v} miss(u))
//   miss'(v) = alpha [v not in S] sum_{u~v} miss(u)
// A warp takes four consecutive rows at a time (one sector of y), two such fours deep, with all the
// loads of a row of up to 32 entries in flight: the step is bound by the chain row pointer -> index ->
// gather, then by the gathers' L2 sectors. Neighbouring fours go to different blocks, because callers'
// graphs often list their hubs first. Rows above kNaHub entries come after the others: a warp each,
// eight gathers per lane in flight, and above kNaChunk entries gathered by the whole block into shared
// memory and added up by one warp, so that no group walks a hub alone. Block b writes its sum of
// hit'(v) to slots[b]. Barabasi-Albert, n = 10^6, m = 8 (88 MB in and out, 16 M gathers): 135 us; a
// warp per row, 256 rows in sequence, took 2,230 us, and blocks of consecutive rows 380 us. Entry positions
// are unsigned: up to 2^31 entries, and what is added to look past a row's end must not wrap.
__global__ void __launch_bounds__(kThreads) na_step(const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                                   int32_t n, int32_t iters, const uint32_t* __restrict__ mask,
                                                   const float2* __restrict__ x, float2* __restrict__ y, float alpha,
                                                   double* __restrict__ slots) {
  __shared__ float2 stage[2][kNaChunk];
  __shared__ uint16_t hubs[kNaMaxHubs], order[kNaMaxHubs];
  __shared__ int n_hubs;
  __shared__ double sums[kNaWarps];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x == 0) n_hubs = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gl = lane & (kNaLanes - 1), grp = lane / kNaLanes;
  // the row at a block's place: (iteration, warp, group)
  auto row_at = [&](int place) {
    return (static_cast<int64_t>(place / kNaGroups) * gridDim.x + blockIdx.x) * kNaGroups + place % kNaGroups;
  };
  double cs = 0.0;
  for (int it = 0; it < iters; it += 2) {
    int64_t r[2];
    int32_t e0[2], e1[2];
    int32_t id[2][4];
    Part p[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int place = ((it + k) * kNaWarps + warp) * kNaGroups + grp;
      r[k] = row_at(place);
      e0[k] = e1[k] = 0;
      if (it + k >= iters) r[k] = n;
      if (r[k] < n) {
        e0[k] = __ldg(rp + r[k]);
        e1[k] = __ldg(rp + r[k] + 1);
      }
      if (e1[k] - e0[k] > kNaHub) {
        if (gl == 0) hubs[atomicAdd(&n_hubs, 1)] = static_cast<uint16_t>(place);
        r[k] = n;  // not ours
        e1[k] = e0[k];
      }
      p[k].zero();
    }
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t j = static_cast<uint32_t>(e0[k]) + q * kNaLanes + gl;
        id[k][q] = j < static_cast<uint32_t>(e1[k]) ? __ldg(ci + j) : -1;
      }
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (id[k][q] >= 0) p[k].add(q, __ldg(x + id[k][q]));
#pragma unroll
    for (int k = 0; k < 2; ++k) {  // entries 32.. of rows longer than that
      const uint32_t end = static_cast<uint32_t>(e1[k]);
      for (uint32_t j0 = static_cast<uint32_t>(e0[k]) + 32; j0 < end; j0 += 32) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t j = j0 + q * kNaLanes + gl;
          if (j < end) p[k].add(q, __ldg(x + __ldg(ci + j)));
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float2 t = p[k].total();
      if (gl == 0 && r[k] < n) cs += na_store(mask, y, r[k], alpha, t.x, t.y);
    }
  }
  __syncthreads();
  // hubs by increasing row, so that the FP64 sum's order does not depend on the atomics
  const int nh = n_hubs;
  for (int a = threadIdx.x; a < nh; a += kThreads) {
    int rank = 0;
    for (int c = 0; c < nh; ++c) rank += hubs[c] < hubs[a];
    order[rank] = hubs[a];
  }
  __syncthreads();
  double hub_cs = 0.0;
  for (int i = warp; i < nh; i += kNaWarps) {
    const int64_t r = row_at(order[i]);
    const int32_t e0 = __ldg(rp + r), e1 = __ldg(rp + r + 1);
    if (e1 - e0 > kNaChunk) continue;
    float sh = 0.0f, sm = 0.0f;
    constexpr int U = 8;
    for (int64_t j0 = e0 + lane; j0 < e1; j0 += 32 * U) {
      int32_t id[U];
      float2 v[U];
#pragma unroll
      for (int k = 0; k < U; ++k) id[k] = j0 + 32 * k < e1 ? __ldg(ci + j0 + 32 * k) : -1;
#pragma unroll
      for (int k = 0; k < U; ++k) v[k] = id[k] >= 0 ? __ldg(x + id[k]) : make_float2(0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k < U; ++k) {
        sh += v[k].x;
        sm += v[k].y;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sh += __shfl_xor_sync(0xffffffffu, sh, o);
      sm += __shfl_xor_sync(0xffffffffu, sm, o);
    }
    if (lane == 0) hub_cs += na_store(mask, y, r, alpha, sh, sm);
  }
  for (int i = 0; i < nh; ++i) {
    const int64_t r = row_at(order[i]);
    const int32_t e0 = __ldg(rp + r), e1 = __ldg(rp + r + 1);
    if (e1 - e0 <= kNaChunk) continue;  // uniform in the block
    float sh = 0.0f, sm = 0.0f;
    constexpr int per = kNaChunk / kThreads;
    float2 v[per];
    auto fetch = [&](int64_t c0) {
#pragma unroll
      for (int k = 0; k < per; ++k) {
        const int64_t j = c0 + k * kThreads + threadIdx.x;
        v[k] = j < e1 ? __ldg(x + __ldg(ci + j)) : make_float2(0.0f, 0.0f);
      }
    };
    fetch(e0);
    int buf = 0;
    for (int64_t c0 = e0; c0 < e1; c0 += kNaChunk, buf ^= 1) {
#pragma unroll
      for (int k = 0; k < per; ++k) stage[buf][k * kThreads + threadIdx.x] = v[k];
      __syncthreads();
      if (c0 + kNaChunk < e1) fetch(c0 + kNaChunk);
      if (warp == 0) {
        const int len = static_cast<int>(min(int64_t(kNaChunk), e1 - c0));
#pragma unroll 8
        for (int k = lane; k < len; k += 32) {
          sh += stage[buf][k].x;
          sm += stage[buf][k].y;
        }
      }
    }
    if (warp == 0) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        sh += __shfl_xor_sync(0xffffffffu, sh, o);
        sm += __shfl_xor_sync(0xffffffffu, sm, o);
      }
      if (lane == 0) hub_cs += na_store(mask, y, r, alpha, sh, sm);
    }
    __syncthreads();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cs += __shfl_xor_sync(0xffffffffu, cs, o);
  if (lane == 0) sums[warp] = cs + hub_cs;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kNaWarps; ++w) t += sums[w];
    slots[blockIdx.x] = t;
  }
}

// out = sum of slots[0..count) in a fixed order (one CTA). Launched as a programmatic dependent.
__global__ void __launch_bounds__(1024) na_reduce(const double* __restrict__ slots, int32_t count,
                                                 double* __restrict__ out) {
  __shared__ double sm[32];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  double v = 0.0;
#pragma unroll 8
  for (int i = threadIdx.x; i < count; i += 1024) v += __ldcg(slots + i);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = sm[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) *out = v;
  }
}

// Device address of the scratch array on the current device; looked up once per device.
gedwalk_status na_scratch(double** out) {
  int dev = 0;
  GW_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNaMaxDevices) return fail(GEDWALK_ERR_INVALID, "device %d not supported", dev);
  std::lock_guard<std::mutex> lk(g_na_mu);
  if (!g_na_ptr[dev]) {
    double* p = nullptr;
    GW_CUDA(cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_na_slots));
    g_na_ptr[dev] = p;
  }
  *out = g_na_ptr[dev];
  return GEDWALK_OK;
}

}  // namespace
}  // namespace gw

using namespace gw;

extern "C" gedwalk_status gedwalk_score_step_noalloc(const int32_t* d_row_ptr, const int32_t* d_col_idx, int32_t n,
                                                     const uint32_t* d_mask, const float* d_x, float* d_y,
                                                     double alpha, double* d_hit_sum, int64_t stream) {
  if (!d_row_ptr || !d_col_idx || !d_mask || !d_x || !d_y || !d_hit_sum)
    return fail(GEDWALK_ERR_INVALID, "gedwalk_score_step_noalloc: a device pointer is NULL");
  if (n < 1 || int64_t(n) > kNaMaxRows)
    return fail(GEDWALK_ERR_INVALID,
                "gedwalk_score_step_noalloc: n = %d outside [1, %lld]: its fixed scratch holds partial sums for "
                "at most %lld rows",
                n, static_cast<long long>(kNaMaxRows), static_cast<long long>(kNaMaxRows));
  if (!(alpha > 0.0)) return fail(GEDWALK_ERR_INVALID, "gedwalk_score_step_noalloc: alpha must be positive");
  if ((reinterpret_cast<uintptr_t>(d_x) | reinterpret_cast<uintptr_t>(d_y) | reinterpret_cast<uintptr_t>(d_hit_sum)) &
      7u)
    return fail(GEDWALK_ERR_INVALID, "gedwalk_score_step_noalloc: x, y and hit_sum must be 8-byte aligned");
  double* slots = nullptr;
  GW_TRY(na_scratch(&slots));
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // iterations of a block (32 rows each): one on small graphs, so that every SM gets some rows; 64 on
  // the largest
  const int64_t steps = (int64_t(n) + kNaRowStep - 1) / kNaRowStep;
  const int32_t iters = static_cast<int32_t>((steps + kNaMaxBlocks - 1) / kNaMaxBlocks);
  const int blocks = static_cast<int>((steps + iters - 1) / iters);
  na_step<<<blocks, kThreads, 0, s>>>(d_row_ptr, d_col_idx, n, iters, d_mask, reinterpret_cast<const float2*>(d_x),
                                      reinterpret_cast<float2*>(d_y), static_cast<float>(alpha), slots);
  GW_KCHECK();
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3(1024);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  GW_CUDA(cudaLaunchKernelEx(&cfg, na_reduce, static_cast<const double*>(slots), static_cast<int32_t>(blocks), d_hit_sum));
  GW_KCHECK();
  return GEDWALK_OK;
}
