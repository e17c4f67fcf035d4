// Device helpers shared by the kernels: per-lane column sums, the best-16 lists of the selection
// passes, stochastic greedy's draw.
#pragma once

#include <cuda_runtime.h>

#include <climits>
#include <cstdint>

namespace gw {

// Pairs of FP32 values hi + lo, |lo| about 2^-24 |hi|: values and sums to about 2^-46 where a GB300's FP64
// units would take 64 times as long. Exact sum and product of two floats (Knuth; Dekker, with fma):
__device__ __forceinline__ float two_sum(float a, float b, float* err) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  *err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
  return s;
}
__device__ __forceinline__ float two_prod(float a, float b, float* err) {
  const float p = __fmul_rn(a, b);
  *err = __fmaf_rn(a, b, -p);
  return p;
}
struct Pair {
  float hi, lo;
  __device__ __forceinline__ void add(float x) {
    float e;
    hi = two_sum(hi, x, &e);
    lo = __fadd_rn(lo, e);
  }
  __device__ __forceinline__ void add(const Pair& x) {
    float e;
    hi = two_sum(hi, x.hi, &e);
    lo = __fadd_rn(lo, __fadd_rn(e, x.lo));
  }
  __device__ __forceinline__ void sub(const Pair& x) { add(Pair{-x.hi, -x.lo}); }
  __device__ __forceinline__ Pair times(const Pair& x) const {
    float e;
    const float p = two_prod(hi, x.hi, &e);
    return Pair{p, __fmaf_rn(hi, x.lo, __fmaf_rn(lo, x.hi, e))};
  }
  __device__ __forceinline__ Pair times(float x) const {
    float e;
    const float p = two_prod(hi, x, &e);
    return Pair{p, __fmaf_rn(lo, x, e)};
  }
  // at least 0: differences of rounded values that would be >= 0 exactly
  __device__ __forceinline__ Pair pos() const { return __fadd_rn(hi, lo) > 0.0f ? *this : Pair{0.0f, 0.0f}; }
  __device__ __forceinline__ double get() const { return static_cast<double>(hi) + static_cast<double>(lo); }
  __device__ __forceinline__ float rounded() const { return __fadd_rn(hi, lo); }
  __device__ __forceinline__ Pair from_lane_xor(int o) const {
    return Pair{__shfl_xor_sync(0xffffffffu, hi, o), __shfl_xor_sync(0xffffffffu, lo, o)};
  }
};
// The same interface in FP64, for kernels of either precision: Wide<T> holds what must not be rounded to T
// when T is FP32.
struct Double {
  double v;
  __device__ __forceinline__ void add(double x) { v += x; }
  __device__ __forceinline__ void add(const Double& x) { v += x.v; }
  __device__ __forceinline__ void sub(const Double& x) { v -= x.v; }
  __device__ __forceinline__ Double times(const Double& x) const { return Double{v * x.v}; }
  __device__ __forceinline__ Double times(double x) const { return Double{v * x}; }
  __device__ __forceinline__ Double pos() const { return Double{v > 0.0 ? v : 0.0}; }
  __device__ __forceinline__ double get() const { return v; }
  __device__ __forceinline__ double rounded() const { return v; }
  __device__ __forceinline__ Double from_lane_xor(int o) const { return Double{__shfl_xor_sync(0xffffffffu, v, o)}; }
};
template <typename T>
struct WideOf {
  using type = Double;
  __device__ __forceinline__ static Double make(double hi, double) { return Double{hi}; }
  __device__ __forceinline__ static Double inverse(double x) { return Double{1.0 / x}; }
  // a + x, the rounding error added to lo
  __device__ __forceinline__ static void accumulate(double& a, double&, double x) { a += x; }
};
template <>
struct WideOf<float> {
  using type = Pair;
  __device__ __forceinline__ static Pair make(float hi, float lo) { return Pair{hi, lo}; }
  __device__ __forceinline__ static Pair inverse(float x) {
    const float r = 1.0f / x;
    return Pair{r, __fmul_rn(r, __fmaf_rn(-x, r, 1.0f))};
  }
  __device__ __forceinline__ static void accumulate(float& a, float& lo, float x) {
    float e;
    a = two_sum(a, x, &e);
    lo = __fadd_rn(lo, e);
  }
};
template <typename T>
using Wide = typename WideOf<T>::type;

__device__ __forceinline__ Pair to_pair(double x) {
  const float hi = static_cast<float>(x);
  return Pair{hi, static_cast<float>(x - static_cast<double>(hi))};
}

// Per-lane column sums over the rows of one unit. FP64 vectors sum in FP64. FP32 vectors sum with
// compensated FP32 additions (Kahan: the error is at most 2u * sum |y| + O(m u^2), u = 2^-24, over a
// unit's m <= 128 rows) and convert once per unit to FP64, in which every later sum (over lanes, units and
// sweeps) is taken. On a GB300 an FP64 addition costs about 64 FP32 ones, and one conversion and
// one FP64 addition per row and column cost more than the rest of the epilogue.
template <typename T, int N>
struct ColAcc {
  double s[N];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int k = 0; k < N; ++k) s[k] = 0.0;
  }
  __device__ __forceinline__ void add(int k, double y) { s[k] += y; }
  __device__ __forceinline__ double get(int k) const { return s[k]; }
};
template <int N>
struct ColAcc<float, N> {
  float s[N], c[N];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int k = 0; k < N; ++k) s[k] = c[k] = 0.0f;
  }
  __device__ __forceinline__ void add(int k, float y) {
    const float t1 = __fsub_rn(y, c[k]);
    const float t = __fadd_rn(s[k], t1);
    c[k] = __fsub_rn(__fsub_rn(t, s[k]), t1);
    s[k] = t;
  }
  __device__ __forceinline__ double get(int k) const { return static_cast<double>(s[k]) - static_cast<double>(c[k]); }
};

// ---------------------------------------------------------------- selection
constexpr int kTopK = 16;

struct Stale {
  float ub;      // last exact gain rounded up (an upper bound for every later step)
  int32_t step;  // step in which it was evaluated, -1 if never
};

constexpr unsigned long long kNoZero = ~0ull;
__host__ __device__ inline int32_t zero_caller(unsigned long long z) {
  return z == kNoZero ? INT_MAX : static_cast<int32_t>(z >> 32);
}
__host__ __device__ inline int32_t zero_internal(unsigned long long z) {
  return static_cast<int32_t>(z & 0xffffffffull);
}

__device__ __forceinline__ bool better(float a, int ia, float b, int ib) { return a > b || (a == b && ia < ib); }

// Stochastic greedy's counter-based draw: the first output of splitmix64 (Steele, Lea & Flood,
// 2014) started from state seed ^ (step << 32) ^ v, v a caller id.
__device__ __forceinline__ uint64_t sample_hash(uint64_t seed, uint32_t step, uint32_t v) {
  uint64_t z = (seed ^ (static_cast<uint64_t>(step) << 32) ^ static_cast<uint64_t>(v)) + 0x9e3779b97f4a7c15ULL;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}

constexpr unsigned kFullMask = 0xffffffffu;

// A warp's sorted list of its kTopK best (value, id) pairs in the order of `better`: lane i <
// kTopK holds the i-th entry (value -1, id INT_MAX: empty); `tag` travels with its entry.
struct WarpList {
  float v = -1.0f;
  int id = INT_MAX;
  int tag = 0;
};

// One compare-exchange step of a bitonic network: the lane keeps the better or the worse of its own
// entry and that of lane ^ j.
__device__ __forceinline__ void list_exchange(float& v, int& id, int& tag, int j, bool keep_better) {
  const float ov = __shfl_xor_sync(kFullMask, v, j);
  const int oi = __shfl_xor_sync(kFullMask, id, j);
  const int ot = __shfl_xor_sync(kFullMask, tag, j);
  if (better(ov, oi, v, id) == keep_better && oi != id) {
    v = ov;
    id = oi;
    tag = ot;
  }
}

// Offers every lane's (x, ix, tag) where `want` holds. Only the lanes that beat the list's last
// entry go in: a few of them one at a time (lowest lane first; after each insertion the others are
// checked again against the new last entry), many of them by sorting the 32 offers (15 steps) and
// merging the best 16 with the list (5 steps). An insertion costs about as much as three of those
// steps, and a warp's first offers would take some thirty. Ids must be distinct. All 32 lanes take
// part.
__device__ __forceinline__ void warp_list_offer(WarpList& w, bool want, float x, int ix, int tag) {
  const int lane = threadIdx.x & 31;
  float tv = __shfl_sync(kFullMask, w.v, kTopK - 1);
  int ti = __shfl_sync(kFullMask, w.id, kTopK - 1);
  const bool enters = want && better(x, ix, tv, ti);
  unsigned m = __ballot_sync(kFullMask, enters);
  if (__popc(m) > 5) {
    float v = enters ? x : -1.0f;
    int id = enters ? ix : INT_MAX, tg = tag;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
      for (int j = k >> 1; j > 0; j >>= 1) list_exchange(v, id, tg, j, ((lane & j) == 0) == ((lane & k) == 0));
    // the best of list[i] and offer[15 - i] are the best 16 of both, a bitonic sequence
    const int src = (kTopK - 1 - lane) & 31;
    const float rv = __shfl_sync(kFullMask, v, src);
    const int ri = __shfl_sync(kFullMask, id, src);
    const int rt = __shfl_sync(kFullMask, tg, src);
    if (lane < kTopK && better(rv, ri, w.v, w.id)) {
      w.v = rv;
      w.id = ri;
      w.tag = rt;
    }
#pragma unroll
    for (int j = kTopK / 2; j > 0; j >>= 1) list_exchange(w.v, w.id, w.tag, j, (lane & j) == 0);
    return;
  }
  while (m) {
    const int src = __ffs(m) - 1;
    const float cv = __shfl_sync(kFullMask, x, src);
    const int ci = __shfl_sync(kFullMask, ix, src);
    const int ct = __shfl_sync(kFullMask, tag, src);
    // the entries ahead of the new one form a prefix of the sorted list
    const int pos = __popc(__ballot_sync(kFullMask, lane < kTopK && better(w.v, w.id, cv, ci)));
    const float uv = __shfl_up_sync(kFullMask, w.v, 1);
    const int ui = __shfl_up_sync(kFullMask, w.id, 1);
    const int ut = __shfl_up_sync(kFullMask, w.tag, 1);
    if (lane == pos) {
      w.v = cv;
      w.id = ci;
      w.tag = ct;
    } else if (lane > pos && lane < kTopK) {
      w.v = uv;
      w.id = ui;
      w.tag = ut;
    }
    tv = __shfl_sync(kFullMask, w.v, kTopK - 1);
    ti = __shfl_sync(kFullMask, w.id, kTopK - 1);
    m &= m - 1;
    m &= __ballot_sync(kFullMask, want && better(x, ix, tv, ti));
  }
}

}  // namespace gw
