// Greedy GED-Walk maximisation (problem (ii), Def. ged-max; Prop. greedy_approx) and
// all-vertex exact marginal gains, on runs of half the walk length (run.cu).
//
// A chain run carries the next steps' guessed winners c_1..c_D, each under S and the earlier ones, and
// brings for every level the best upper bounds of the unevaluated vertices and the exact gain of its
// guess. A step takes the guess once no bound (inflated by the rounding tolerance) reaches its gain;
// otherwise the best-bounded vertices are evaluated exactly, side by side under S, until the best
// exact gain is beyond every bound. No result depends on the guesses. A vertex whose bound is exactly
// 0 has gain exactly 0. Among equal gains the lowest caller id wins.
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

struct Cand {
  double g;
  int32_t v;       // internal id
  int32_t caller;  // caller id
};
// exact-gain order: larger gain first, then the lower caller id
bool cand_before(const Cand& a, const Cand& b) { return a.g > b.g || (a.g == b.g && a.caller < b.caller); }

}  // namespace

gedwalk_status greedy_shape(const Graph& g, const Resolved& r, int32_t flags, GreedyShape* out) {
  GreedyShape sh{};
  const bool adaptive = (flags & GEDWALK_ADAPTIVE_L) != 0;
  sh.ell_max = 1;
  while (adaptive && sh.ell_max < r.L) sh.ell_max *= 2;
  const int32_t tab_L = adaptive ? sh.ell_max : r.L;
  // One-step runs (lookahead off, spec_cols): phi^miss and the candidates likely to win. One certifies
  // most steps (a miss costs one candidate batch).
  sh.cols_fused = 2;
  if (r.spec_cols != 0) {
    if (!(r.spec_cols == 2 || r.spec_cols == 4 || (r.spec_cols == 8 && !r.fp64)))
      return fail(GEDWALK_ERR_INVALID, "spec_cols must be 0, 2, 4 or (FP32) 8");
    sh.cols_fused = r.spec_cols;
  }
  // Lookahead: one run carries `levels` steps, level d under S + {c_1..c_d} with
  // the guessed winners c_d; a step whose winner was guessed needs no run of its own. The run's rows
  // hold levels + 1 columns. A gather costs one L2 sector request whatever the row width up to 32
  // bytes, so 7 FP32 levels cost little more per sweep than one.
  const bool plain = (flags & (GEDWALK_ADAPTIVE_L | GEDWALK_STOCHASTIC | GEDWALK_GAINS_ALL)) == 0;
  sh.levels = 1;
  if (!(flags & GEDWALK_GAINS_ALL)) {
    // FP64: 64-byte rows, two sectors a gather, but seven steps for them: a sweep of 8 columns takes
    // 456 us instead of 270 on Barabasi-Albert n = 10^6 (k = 25: 9.2 -> 7.4 ms).
    sh.levels = run_width(g, tab_L, 8, r.fp64) - 1;
    if (plain && !g.directed && r.lookahead != 0) {
      if (!(r.lookahead == 1 || r.lookahead == 3 || (!r.fp64 && r.lookahead == 7)))
        return fail(GEDWALK_ERR_INVALID, "lookahead must be 0, 1, 3 or (FP32) 7");
      sh.levels = r.lookahead;
    }
    if ((!plain || g.directed) && r.spec_cols != 0) sh.levels = 1;  // the caller fixed the one-step width
  }
  // Candidate batches run when the evaluated guess is not certified: as wide as the chains.
  sh.cols_cand = run_width(g, tab_L, 8, r.fp64);
  sh.cols_all = run_width(g, tab_L, r.fp64 ? 8 : 16, r.fp64);
  if (r.max_cols > 0) {
    sh.levels = std::min(sh.levels, r.max_cols - 1);
    for (int32_t* c : {&sh.cols_fused, &sh.cols_cand, &sh.cols_all}) *c = std::min(*c, r.max_cols);
  }
  sh.tab_L = tab_L;
  sh.cols_max = std::max({sh.levels > 1 ? sh.levels + 1 : sh.cols_fused, sh.cols_cand,
                          (flags & GEDWALK_GAINS_ALL) ? sh.cols_all : 0, 2});
  *out = sh;
  return GEDWALK_OK;
}

gedwalk_status ensure_run_tables(Graph& g, Workspace& ws, const Resolved& r, const GreedyShape& sh, int32_t flags) {
  const bool adaptive = (flags & GEDWALK_ADAPTIVE_L) != 0;
  if (adaptive) GW_TRY(ensure_totals(g, r.alpha, sh.ell_max + 1, r.stream));
  if (!g.directed || g.n_active == 0 || (flags & GEDWALK_GAINS_ALL)) return GEDWALK_OK;
  const int32_t rows = walk_rows(g, (adaptive ? sh.ell_max : r.L) + 1);
  {
    std::shared_lock<std::shared_mutex> rl(g.tt_lock);
    if (g.tt_alpha != r.alpha || g.tt_rows < rows) return GEDWALK_OK;
  }
  return ensure_totals_fwd(g, ws, r.alpha, rows, r.stream);
}

int64_t maximize_footprint(const Graph& g, const Resolved& r, int32_t flags, int32_t k) {
  GreedyShape sh{};
  if (greedy_shape(g, r, flags, &sh) != GEDWALK_OK) return 0;
  const int64_t n = g.n, es = r.fp64 ? 8 : 4;
  int64_t b = run_bytes(g, sh.tab_L, sh.cols_max, r.fp64, (flags & GEDWALK_GAINS_ALL) == 0);
  if ((flags & GEDWALK_GAINS_ALL) && small_gain_cols(g, r.fp64) > 0)  // one launch's table, vectors and gains
    b += n * (es * ((sh.tab_L + 1) / 2 + 3) + 8) + static_cast<int64_t>(std::max(g.plan.num_slots, 1)) * 8;
  // (directed: the sums of the walk totals; adaptive: the final group is scored)
  if (g.directed) b += static_cast<int64_t>(std::max(std::max(g.plan.num_slots, g.plan_r.num_slots), 1)) * 2 * 8;
  if (g.directed && (flags & GEDWALK_ADAPTIVE_L)) b += 2 * n * 2 * es;
  return b + 4 * (static_cast<int64_t>(k) + 1);
}

namespace {
// What the loop needs to know of a maximisation.
struct GreedyRun {
  int32_t k;
  int32_t flags;
  GreedyShape shape;
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

// The greedy loop.
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
  // Relative inflation of bounds against the rounding of the values a certification compares, beyond what
  // the bounds themselves allow for: four times one sweep's (run.h) for up to four of them, and like the root
  // of their number beyond, as the bounds' own slack (run.cu). More costs runs where gains lie close: R-MAT
  // scale 22, k = 100 takes 35.5 ms with 1e-6, 39.8 with 3e-6 and 55 to 66 with 1e-5 (1, 3 and 10 of 100 steps
  // not certified by their guess), and 37.8 with four times the bounds' own slack; l-doubling there, 7 sweeps a
  // run, 62.9 ms where the tolerance grew with their number; the other graphs measured do not care.
  auto tol = [&]() {
    return r.fp64 ? 1e-11 : 4.0 * sweep_rounding<float>() * std::sqrt(std::max(1.0, 0.25 * (eng.H - 1)));
  };
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
  // FP64 rows of 8 columns cost more than rows of 4 in every sweep, so they wait for a chain that held
  // for three steps (on a small graph one winner changes the order of the next ones) and are no use for
  // three steps or fewer. k = 20, ms starting with three / seven: Erdos-Renyi 4,000 1.38 / 1.61, 12,000
  // 1.19 / 1.38, 30,000 1.72 / 2.08, 100,000 3.51 / 2.99, 400,000 9.55 / 8.11; Barabasi-Albert 4,000 0.60 /
  // 0.49, 30,000 0.76 / 0.64, 400,000 2.73 / 2.33; R-MAT of 2^13 rows 0.85 / 1.10, 2^18 2.87 / 2.43. So the line
  // could lie anywhere between 12,000 and 100,000, and hubs would have it lower. Waiting for one or two steps
  // instead of three changes nothing, for five costs up to a half more.
  const bool two_widths = r.fp64 && sh.levels == 7;
  int width = two_widths && (g.n_active < 20000 || p.k <= 3) ? 3 : n_spec;
  int held = -1;                // steps the last chain has carried (-1: none yet)
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
        eng.sweeps += eng.H;  // of phi^miss; the columns' steps are no sweeps
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
          if (two_widths && held >= 0) width = held >= 3 ? 7 : 3;
          held = 0;
          look_c = spec;
          look_c.resize(width, -1);
          draws(step);
          GW_TRY(eng.run(chain, width + 1, true, look_c));
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
          const double ub0 = top.empty() ? -1.0 : static_cast<double>(sel.val[0]) * (1.0 + tol());
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
          // rows of four columns for the first batch where the chain's are; more candidates at a time after it
          const int cols_cand = two_widths && width == 3 && first_batch ? 4 : sh.cols_cand;
          first_batch = false;
          std::vector<int32_t> last(top.begin(), top.begin() + std::min<size_t>(top.size(), cols_cand - 1));
          draws(step);
          if (everyone) eng.in->thr[0] = ~0ull;
          GW_TRY(eng.run(false, cols_cand, true, last));
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
      const bool taken = chain && best.v == look_c[lvl];
      held += taken;
      if (taken && lvl + 1 < width && look_c[lvl + 1] >= 0) ++lvl;
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
    GW_TRY(ensure_run_tables(g, ws, r, p.shape, flags));
    std::shared_lock<std::shared_mutex> rl(g.tt_lock);
    if (g.tt_alpha != r.alpha || static_cast<int32_t>(g.Wa.size()) < p.shape.ell_max + 1)
      return fail(GEDWALK_ERR_INVALID, "the walk-total table was replaced for another alpha during the call");
    p.Wa.assign(g.Wa.begin(), g.Wa.begin() + p.shape.ell_max + 1);
  }
  std::vector<int32_t> S_all;
  for (;;) {
    ws.st_evals = ws.st_batches = ws.st_sweeps = ws.st_spec_miss = ws.st_sep_fail = 0;
    ws.st_ell.clear();
    const gedwalk_status st = maximize_runs(g, ws, r, p, init_int, group, gains, &S_all);
    if (st == GEDWALK_OK) break;
    if (st != GEDWALK_ERR_OOM || p.shape.cols_max <= 2) return st;
    // the device cannot hold rows this wide: again with half the columns (the results do not depend on them)
    GW_CUDA(cudaStreamSynchronize(r.stream));
    r.max_cols = p.shape.cols_max / 2;
    GW_TRY(greedy_shape(g, r, flags, &p.shape));
  }
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
  int cols_all = run_width(g, r.L, r.fp64 ? 8 : 16, r.fp64);
  std::vector<char> inS(g.n, 0);
  for (int32_t v : S_int) inS[v] = 1;
  for (int32_t v = 0; v < g.n; ++v) gains_caller[v] = 0.0;  // an isolated vertex gains nothing
  if (small_gain_cols(g, r.fp64) > 0) {
    std::vector<double> got(g.n_active);
    GW_TRY(small_gains(g, ws, r, S_int, got.data()));
    for (int32_t v = 0; v < g.n_active; ++v) gains_caller[g.perm[v]] = got[v];
    guard.ok = true;
    return GEDWALK_OK;
  }
  RunEngine eng(g, ws, r, s);
  for (;; cols_all /= 2) {  // narrower where the device cannot hold the vectors
    const gedwalk_status st = eng.setup(r.L, cols_all, false, S_int);
    if (st == GEDWALK_OK) break;
    if (st != GEDWALK_ERR_OOM || cols_all <= 2) return st;
    GW_CUDA(cudaStreamSynchronize(s));
  }
  GW_TRY(eng.set_length(r.L, false));
  std::vector<int32_t> batch;
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
