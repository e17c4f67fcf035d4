// Runs of sweeps of half the walk length, joined by the meeting pass (run.cu).
#pragma once

#include <cuda_runtime.h>

#include <functional>

#include "device_util.cuh"
#include "internal.h"

namespace gw {

constexpr int kRunCols = 16;            // widest run: column 0 and 15 candidates
constexpr int kRunCands = kRunCols - 1;
constexpr int kRunLevels = 7;           // lookahead levels with a selection of their own
constexpr int kMeetPerSM = 3;           // resident blocks of the meeting pass per SM
constexpr int kMeetBlocks = 152 * kMeetPerSM;

// What a sweep adds to a stored value's relative error. A row's sum takes at most 39 additions one after the
// other, whatever its length (32 in a lane, five over the lanes; hubs' slices are compensated), so
// roundings of u = 2^-24 add up to about sqrt(39) u / 2 = 1.9e-7 (Higham & Mary 2019: sqrt, not 39 u).
// Measured on R-MAT scale 22 (k = 100, rows of up to 160 slices), Erdos-Renyi 100,003 (L = 40) and directed
// R-MAT scale 18: FP32 gains within 1.4e-7 of the FP64 ones after all sweeps, picks the same.
template <typename T>
__host__ __device__ constexpr float sweep_rounding() {
  return sizeof(T) == 8 ? 1e-15f : 2.5e-7f;
}

// What a run is told, copied to the device as its first operation.
struct RunIn {
  int32_t cand[kRunCols];      // candidate of column j + 1, -1: none
  int32_t added[kRunCols];     // vertices that joined S since the last run
  int32_t n_added;
  int32_t n_stale;             // exact gains known on the host, to be recorded
  int32_t stale_id[kRunCols];
  int32_t stale_step[kRunCols];
  double stale_gain[kRunCols];
  int32_t step;                // greedy step of level 0
  uint64_t seed;               // stochastic greedy: the draws of the levels' steps
  uint64_t thr[kRunLevels];    // UINT64_MAX: every vertex takes part
};

// The best kTopK bounds among the vertices not evaluated, for one level.
struct LevelSel {
  float val[kTopK];
  int32_t id[kTopK];
  // the vertex with bound exactly 0 and the smallest caller id, (caller id << 32) | internal id
  unsigned long long zero_min;
  int32_t sampled;  // stochastic greedy: sampled vertices outside the level's set
  int32_t pad;
};

struct RunOut {  // device -> host, one copy per run
  LevelSel lv[kRunLevels];
  double gains[kRunCols];
};

struct RunDev {  // device-side state of the runs of one workspace
  RunIn in;
  RunOut out;
  int32_t live[2][kRunCols];  // per set of vectors: whether candidate j's row has an entry outside its base set
  int32_t adj[2][kRunCols];   // chain: earlier candidates in candidate j's row
  int32_t done;            // blocks of the meeting (or guess) pass that have finished
};

// Runs a launch sequence, captured once per configuration and replayed as a CUDA graph; directly on the
// legacy default stream. The capture comes with the second use, above kLateEntries entries with the
// fourth: sweeps outlast their launches there, so a new graph's short maximisation gains nothing from it.
// First call of k = 10 on a new handle, capture with the second / fourth use, ms: R-MAT scale 20 (31 M
// entries) 1.86 / 1.57, scale 18 (7.6 M) 1.11 / 0.73; Barabasi-Albert 4 to 16 M 1.03 / 0.96 to 1.42 / 1.40;
// below the line 0.52 / 0.64 (R-MAT scale 16) to 0.74 / 0.45 (Barabasi-Albert 1.6 M), within the runs' spread.
// `issue` gets the two timing events of a capture (or null).
constexpr int64_t kLateEntries = int64_t(4) << 20;
struct Sequence {
  uint64_t key;
  int kernels, sweeps;
  double bytes;
  int prof_key;
  int64_t nnz;
};
gedwalk_status run_sequence(Workspace& ws, cudaStream_t s, const Sequence& q,
                            const std::function<gedwalk_status(bool profile, const std::vector<cudaEvent_t>* ev)>& issue);
// The stream a run uses: the caller's, or the workspace's own for the legacy default stream.
gedwalk_status greedy_stream(Workspace& ws, cudaStream_t caller, cudaStream_t* out);
// After a synchronisation: hands the sweep timings of graph replays to the profiler.
void read_graph_timing(Workspace& ws);
uint64_t mix_all(std::initializer_list<uint64_t> vs);

// Stored vectors are kept to about this size: beyond it, and where the device cannot hold them, rows get
// narrower (fewer steps or candidates a run) and scoring keeps a ring of vectors.
constexpr int64_t kWideBytes = int64_t(32) << 30;
// The widest rows of at most `cols` columns, at least 2, whose ceil(L/2) stored vectors stay below it.
inline int run_width(const Graph& g, int32_t L, int cols, bool fp64) {
  const int64_t cell = static_cast<int64_t>(g.n_active) * ((L + 1) / 2) * (g.directed ? 2 : 1) * (fp64 ? 8 : 4);
  while (cols > 2 && cell * cols > kWideBytes) cols /= 2;
  return cols;
}

// The runs of one maximisation (or one gains call).
struct RunEngine {
  Graph& g;
  Workspace& ws;
  const Resolved& r;
  cudaStream_t s;
  int32_t L = 0, H = 0;
  int32_t n_scan = 0;  // rows of the selections (stochastic greedy scans isolated vertices too)
  bool draws = false;  // stochastic greedy: the runs keep the last level's bounds for guess()
  int64_t sweeps = 0;
  RunIn* in = nullptr;   // pinned; step, seed, thr and the stale list are the caller's to fill
  RunOut* out = nullptr; // pinned; valid after run() or guess()
  std::vector<int32_t> added;  // joined S on the host, not yet on the device

  RunEngine(Graph& g_, Workspace& ws_, const Resolved& r_, cudaStream_t s_) : g(g_), ws(ws_), r(r_), s(s_) {}
  // Buffers for runs of up to cols columns and walk length L_max; S = init.
  gedwalk_status setup(int32_t L_max, int cols, bool select, const std::vector<int32_t>& init);
  // Walk length of the following runs; with a selection, the tail bounds for it.
  gedwalk_status set_length(int32_t length, bool select);
  // One run: chain (candidate j under S + the earlier ones) or not (every candidate under S).
  gedwalk_status run(bool chain, int cols, bool select, const std::vector<int32_t>& cand);
  // Selections of `levels` steps' samples from the last pass's bounds (a choice of guesses only).
  gedwalk_status guess(int levels);
  void stale(int32_t v, double gain, int32_t step);

 private:
  template <typename T>
  gedwalk_status own_tails();
  gedwalk_status push_added();
  gedwalk_status issue(bool chain, int cols, bool select, bool profile, const std::vector<cudaEvent_t>* ev);
};

// Device bytes of the buffers RunEngine::setup makes.
int64_t run_bytes(const Graph& g, int32_t L_max, int cols, bool fp64, bool select);

}  // namespace gw
