"""The calls whose speed is watched: what a user of the library has it do, over the sizes it is used at.

Sizes and graph families are those of bench.py, the tests and the serving mix: Erdos-Renyi (long walks,
L about 30), Barabasi-Albert and R-MAT graphs (hubs, L about 9), FP64 and FP32 walk vectors, undirected,
directed and weighted graphs, and the plain, stochastic and l-doubling greedy. Graphs are drawn on the GPU
from the seed alone and uploaded through the public API; the handle is what a program keeps between calls.

A call that asks for FP32 walk vectors gets values of that accuracy, and its program keeps them as float32;
FP64 calls keep float64. Groups, lengths and counters are whole numbers.
"""
import math

import numpy as np
import torch

from paper_1910_13874_gb300 import gedwalk


# ---------------------------------------------------------------------------- graphs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _csr(u, v, n, directed):
    """(row_ptr, col_idx) int32 on the host: no self-loops, no repeats, both directions unless directed."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = u * n + v
    if not directed:
        key = torch.cat([key, v * n + u])
    key = torch.unique(key)
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=key.device)
    row_ptr[1:] = torch.bincount(torch.div(key, n, rounding_mode="floor"), minlength=n).cumsum(0)
    return row_ptr.to(torch.int32).cpu().numpy(), (key % n).to(torch.int32).cpu().numpy()


def _er(n, deg, seed, directed=False):
    g = _gen(seed)
    m = int(round(n * deg / (1 if directed else 2)))
    u = torch.randint(n, (m,), device="cuda", generator=g)
    v = torch.randint(n, (m,), device="cuda", generator=g)
    return _csr(u, v, n, directed)


def _ba(n, m, seed):
    """Preferential attachment: arc i of vertex v copies an endpoint of a uniformly drawn earlier arc."""
    g = _gen(seed)
    arcs = n * m
    src = torch.arange(arcs, device="cuda") // m
    pos = torch.arange(arcs, device="cuda")
    # place 2i holds src[i], place 2i + 1 the content of an earlier place
    ptr = (torch.rand(arcs, device="cuda", generator=g, dtype=torch.float64) * (2 * (src * m)).clamp(min=1)).long()
    dst = torch.full((arcs,), -1, dtype=torch.int64, device="cuda")
    first = pos < m * (m + 1)  # the first vertices attach to each other
    dst[first] = pos[first] % (m + 1)
    cur = ptr.clone()
    todo = torch.nonzero(~first).flatten()
    while todo.numel():
        c = cur[todo]
        even = c % 2 == 0
        dst[todo[even]] = src[torch.div(c[even], 2, rounding_mode="floor")]
        odd = todo[~even]
        i = torch.div(cur[odd], 2, rounding_mode="floor")
        known = dst[i] >= 0
        dst[odd[known]] = dst[i[known]]
        cur[odd[~known]] = ptr[i[~known]]
        todo = odd[~known]
    return _csr(src, dst, n, False)


def _rmat(scale, ef, seed, directed=False):
    g = _gen(seed)
    n, m = 1 << scale, ef << scale
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(scale):  # quadrant probabilities 0.57, 0.19, 0.19, 0.05
        r = torch.rand(m, device="cuda", generator=g)
        u = 2 * u + (r >= 0.76)
        v = 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    p = torch.randperm(n, device="cuda", generator=g)
    return _csr(p[u], p[v], n, directed)


def _graph(case, seed):
    d = bool(case.get("directed"))
    if case["graph"] == "er":
        return _er(case["n"], case["deg"], seed, d)
    if case["graph"] == "ba":
        return _ba(case["n"], case["deg"], seed)
    return _rmat(case["scale"], case["deg"], seed, d)


def _n(case):
    return 1 << case["scale"] if case["graph"] == "rmat" else case["n"]


def _nnz(case):
    """Directed entries of the CSR, but for the repeats an R-MAT or Erdos-Renyi draw drops."""
    per = {"er": case["deg"], "ba": 2 * case["deg"], "rmat": 2 * case["deg"]}[case["graph"]]
    if case.get("directed") and case["graph"] == "rmat":
        per = case["deg"]
    return _n(case) * per


def _groups(case, seed):
    rng = np.random.default_rng([int(seed), 42])
    n = _n(case)
    sizes = rng.integers(1, case["size"] + 1, size=case["groups"])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    mem = np.concatenate([rng.choice(n, size=int(s), replace=False) for s in sizes]).astype(np.int32)
    return off, mem


def _set(case, seed):
    return np.random.default_rng([int(seed), 7]).choice(_n(case), size=case["size"], replace=False).astype(np.int32)


# ---------------------------------------------------------------------------- the cases
def listed():
    return [
        # one recurrence step on the caller's own device buffers: a service that may not allocate
        dict(name="step_ba_1m", kind="step", graph="ba", n=1_000_000, deg=8, size=100),
        # the smallest call: scoring five vertices of a 1000-vertex graph, FP64 (latency, launches)
        dict(name="score_er_1000", kind="score", graph="er", n=1000, deg=10, size=5, prec="fp64", eps=1e-6),
        # scoring one group on a graph with hubs
        dict(name="score_rmat_20", kind="score", graph="rmat", scale=20, deg=16, size=100, prec="fp32", eps=1e-4),
        # many groups at once: the batched-scoring workload at an eighth of its 4096 groups
        dict(name="batch_ba_1m", kind="batch", graph="ba", n=1_000_000, deg=8, groups=512, size=100, prec="fp32",
             eps=1e-4),
        # every vertex's exact gain, as an analysis of a small network asks for (an odd size)
        dict(name="gains_er_3001", kind="gains", graph="er", n=3001, deg=10, size=4, prec="fp32", eps=1e-4),
        # the small maximisation: k = 5 in FP64 (latency)
        dict(name="max_er_1000", kind="max", graph="er", n=1000, deg=10, k=5, prec="fp64", eps=1e-6),
        # a request of the serving mix: long walks, many gains close together
        dict(name="max_er_100k", kind="max", graph="er", n=100_003, deg=16, k=27, prec="fp32", eps=1e-4),
        # FP64 walk vectors at the Barabasi-Albert benchmark's size
        dict(name="max_ba_1m_fp64", kind="max", graph="ba", n=1_000_000, deg=8, k=25, prec="fp64", eps=1e-4),
        # the headline: greedy k = 100 on R-MAT scale 22
        dict(name="max_rmat_22", kind="max", graph="rmat", scale=22, deg=16, k=100, prec="fp32", eps=1e-4),
        # the paper's lazy greedy with l-doubling (Algorithm 2)
        dict(name="max_rmat_20_doubling", kind="max", graph="rmat", scale=20, deg=16, k=50, prec="fp32", eps=1e-4,
             adaptive=True),
        # a directed graph (two orientations)
        dict(name="max_rmat_18_directed", kind="max", graph="rmat", scale=18, deg=16, k=20, prec="fp32", eps=1e-4,
             directed=True),
        # end to end from host arrays: upload, a short maximisation with its walk totals, release
        dict(name="fresh_rmat_20", kind="fresh", graph="rmat", scale=20, deg=16, k=10, prec="fp32", eps=1e-4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "score", "score", "batch", "gains", "max", "max", "max", "max", "fresh"])
    family = rng.choice(["er", "ba", "rmat"])
    case = {"kind": kind, "graph": family}
    if kind == "gains":
        family = case["graph"] = rng.choice(["er", "ba"])
        case["n"] = _log_int(rng, 300, 4000)
        case["deg"] = rng.choice([6, 8, 10, 16]) if family == "er" else rng.choice([4, 8])
    elif family == "rmat":
        case["scale"] = rng.randint(12, 19)
        case["deg"] = rng.choice([8, 16])
    else:
        case["n"] = _log_int(rng, 1000, 400_000)
        case["deg"] = rng.choice([8, 10, 16, 32]) if family == "er" else rng.choice([4, 8, 16])
    if kind == "step":
        case["size"] = _log_int(rng, 1, 300)
        return case
    case["prec"] = "fp32" if kind == "batch" else rng.choice(["fp32", "fp32", "fp64"])
    case["eps"] = rng.choice([1e-3, 1e-4, 1e-5])
    if kind == "batch":
        case["groups"] = _log_int(rng, 5, 600)
        case["size"] = rng.choice([5, 30, 100])
    elif kind in ("score", "gains"):
        case["size"] = _log_int(rng, 1, 200)
    else:
        case["k"] = _log_int(rng, 2, 40)
    if kind in ("max", "fresh", "score") and rng.random() < 0.5:
        case[rng.choice(["weighted", "directed"] if family != "ba" else ["weighted"])] = True
    if kind == "max" and rng.random() < 0.3:
        case[rng.choice(["adaptive", "stochastic"])] = True
    return case


# ---------------------------------------------------------------------------- a program's state and calls
def _params(case, seed):
    kw = dict(epsilon=case["eps"], precision=case["prec"])
    if case.get("adaptive"):
        kw["adaptive"] = True
    if case.get("stochastic"):
        kw.update(stochastic=True, eta=0.1, seed=int(seed))
    return gedwalk.make_params(**kw)


def prepare(case, seed):
    row_ptr, col_idx = _graph(case, seed)
    if case["kind"] == "step":
        return _prepare_step(case, seed, row_ptr, col_idx)
    state = {"case": case, "params": _params(case, seed)}
    upload = dict(weighted=bool(case.get("weighted")), directed=bool(case.get("directed")))
    if case["kind"] == "fresh":
        state.update(row_ptr=row_ptr, col_idx=col_idx, upload=upload)
        return state
    state["G"] = gedwalk.Graph(row_ptr, col_idx, **upload)
    if case["kind"] == "batch":
        state["groups"] = _groups(case, seed)
    elif case["kind"] in ("score", "gains"):
        state["S"] = _set(case, seed)
    return state


def _step_inputs(case, seed, row_ptr):
    """Mask words, (hit, miss) pairs a few steps into a run, and alpha."""
    n = _n(case)
    S = _set(case, seed)
    words = np.zeros((n + 31) // 32, dtype=np.uint32)
    np.bitwise_or.at(words, S >> 5, np.uint32(1) << (S & 31).astype(np.uint32))
    x = torch.rand(n, 2, device="cuda", generator=_gen(int(seed) + 1))
    x[torch.from_numpy(S).long().cuda(), 1] = 0.0
    return words, x, 1.0 / (1.0 + float(np.diff(row_ptr).max()))


def _prepare_step(case, seed, row_ptr, col_idx):
    words, x, alpha = _step_inputs(case, seed, row_ptr)
    return {"case": case, "row_ptr": torch.from_numpy(row_ptr).cuda(), "col_idx": torch.from_numpy(col_idx).cuda(),
            "mask": torch.from_numpy(words.view(np.int32)).cuda(), "x": x, "y": torch.empty_like(x),
            "hit": torch.zeros(1, dtype=torch.float64, device="cuda"), "alpha": alpha}


def _kept(case, v):
    """Values in the precision the call asked for."""
    t = np.float32 if case["prec"] == "fp32" else np.float64
    return v.astype(t) if isinstance(v, np.ndarray) else t(v)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        n = state["x"].shape[0]
        gedwalk.score_step_noalloc(state["row_ptr"].data_ptr(), state["col_idx"].data_ptr(), n,
                                   state["mask"].data_ptr(), state["x"].data_ptr(), state["y"].data_ptr(),
                                   state["alpha"], state["hit"].data_ptr(),
                                   stream=torch.cuda.current_stream().cuda_stream)
        return {"y": state["y"], "hit": state["hit"]}
    if kind == "score":
        score, L, bound = state["G"].score(state["S"], params=state["params"])
        return {"score": _kept(case, score), "L": L, "bound": bound}
    if kind == "batch":
        scores, L = state["G"].score_batch(*state["groups"], params=state["params"])
        return {"scores": _kept(case, scores), "L": L}
    if kind == "gains":
        gains, L = state["G"].gains(state["S"], params=state["params"])
        return {"gains": _kept(case, gains), "L": L}
    if kind == "max":
        G = state["G"]
        group, gains, score, L = G.maximize(case["k"], params=state["params"])
        out = {"group": group, "gains": _kept(case, gains), "score": _kept(case, score), "L": L}
        if case.get("adaptive"):
            out["lengths"] = G.maximize_lengths()[0]
        return out
    G = gedwalk.Graph(state["row_ptr"], state["col_idx"], **state["upload"])
    group, gains, score, L = G.maximize(case["k"], params=state["params"])
    out = {"nnz": G.nnz, "dmax": G.dmax, "group": group, "gains": _kept(case, gains), "score": _kept(case, score),
           "L": L}
    G.free()
    return out


def work(case):
    """The CSR read once, the other inputs read and the outputs written once; one multiply-add per entry
    for every vertex set whose walks have to be counted (the group, each group, each pick)."""
    n, nnz = _n(case), _nnz(case)
    csr = 4.0 * nnz + 4.0 * (n + 1)
    kind = case["kind"]
    if kind == "step":
        return {"bytes": csr + n / 8 + 16.0 * n + 8, "flops": 2.0 * 2 * nnz}
    if kind == "score":
        return {"bytes": csr + 4 * case["size"] + 20, "flops": 2.0 * nnz}
    if kind == "batch":
        return {"bytes": csr + case["groups"] * (4 * (case["size"] + 1) / 2 + 8.0), "flops": 2.0 * nnz * case["groups"]}
    if kind == "gains":
        return {"bytes": csr + 4 * case["size"] + 8.0 * n, "flops": 2.0 * nnz}
    return {"bytes": csr + 12.0 * case["k"], "flops": 2.0 * nnz * case["k"]}


# ---------------------------------------------------------------------------- 64-bit values
class _Exact:
    """The definitions of the paper in plain torch, 64 bits: walk recurrences on a sparse matrix."""

    def __init__(self, case, seed):
        rp, ci = _graph(case, seed)
        self.case, self.n, self.nnz = case, len(rp) - 1, len(ci)
        deg = np.diff(rp.astype(np.int64))
        rpt, cit = torch.from_numpy(rp.astype(np.int64)).cuda(), torch.from_numpy(ci.astype(np.int64)).cuda()
        rows = torch.repeat_interleave(torch.arange(self.n, device="cuda"), torch.from_numpy(deg).cuda())
        w = torch.ones(self.nnz, dtype=torch.float64, device="cuda")
        self.dmax = int(deg.max())
        self.delta = float(self.dmax)
        if case.get("weighted"):
            s = torch.from_numpy(np.where(deg > 0, 1.0 / np.sqrt(np.maximum(deg, 1)), 0.0)).cuda()
            w = s[rows] * s[cit]
            self.delta = float(torch.zeros(self.n, dtype=torch.float64, device="cuda").index_add_(0, rows, w).max())
        self.A = torch.sparse_csr_tensor(rpt, cit, w, (self.n, self.n))
        self.At = self.A
        if case.get("directed"):
            ind = torch.bincount(cit, minlength=self.n)
            self.delta = float(min(self.dmax, int(ind.max())))
            order = torch.sort(cit * self.n + rows).indices
            rpr = torch.zeros(self.n + 1, dtype=torch.int64, device="cuda")
            rpr[1:] = ind.cumsum(0)
            self.At = torch.sparse_csr_tensor(rpr, rows[order], w[order], (self.n, self.n))
        self.alpha = 1.0 / (1.0 + self.delta)

    def length(self, eps):
        """(L, B_L, [B_0 ..]): the first l >= 1 whose combinatorial tail bound is below eps."""
        coef = self.alpha * self.delta / (1.0 - self.alpha * self.delta)
        x = torch.ones(self.n, dtype=torch.float64, device="cuda")
        B = [coef * self.n]
        while len(B) < 2 or not B[-1] < eps:
            x = self.alpha * (self.A @ x)
            B.append(coef * float(x.sum()))
        return len(B) - 1, B[-1], B

    def _mask(self, S):
        m = torch.ones(self.n, dtype=torch.float64, device="cuda")
        m[torch.as_tensor(np.asarray(S, dtype=np.int64)).cuda()] = 0.0
        return m

    def scores(self, groups, L):
        """GED_{<=L} of each group by the two-state recurrence, the groups as columns."""
        out = []
        wide = max(1, min(len(groups), int(2e9 // (self.n * 32))))
        for a in range(0, len(groups), wide):
            M = torch.stack([self._mask(S) for S in groups[a:a + wide]], 1)
            h, m = 1.0 - M, M.clone()
            tot = torch.zeros(M.shape[1], dtype=torch.float64, device="cuda")
            for _ in range(L):
                ah, am = self.alpha * (self.A @ h), self.alpha * (self.A @ m)
                h, m = ah + (1.0 - M) * am, M * am
                tot += h.sum(0)
            out.append(tot)
        return torch.cat(out).cpu().numpy()

    def table(self, mask, L, A):
        rows = [mask]
        for _ in range(L):
            rows.append(mask * (self.alpha * (A @ rows[-1])))
        return torch.stack(rows)

    def columns(self, mask, phi, cand):
        """Exact gains of cand: walks that avoid S, through the candidate."""
        c, j = torch.as_tensor(cand, device="cuda"), torch.arange(len(cand), device="cuda")
        h = torch.zeros(self.n, len(cand), dtype=torch.float64, device="cuda")
        h[c, j] = 1.0
        tot = torch.zeros(len(cand), dtype=torch.float64, device="cuda")
        for t in range(1, phi.shape[0]):
            h = mask[:, None] * (self.alpha * (self.A @ h))
            h[c, j] = phi[t][c]
            tot += h.sum(0)
        return tot.cpu().numpy()

    def best(self, S, L, need, stale, allowed=None):
        """[(gain, vertex)] best first: at least `need` values above every other vertex's bound."""
        mask = self._mask(S)
        phi = self.table(mask, L, self.A)
        psi = self.table(mask, L, self.At) if self.case.get("directed") else phi
        Q = psi.cumsum(0)
        ub = (phi[0] * (Q[L] - psi[0]) + sum(phi[a] * Q[L - a] for a in range(1, L + 1))).cpu().numpy()
        ub = np.minimum(ub, stale)
        ub[list(S)] = -1.0
        if allowed is not None:
            ub[~allowed] = -1.0
        got = {}
        while True:
            order = np.argpartition(-ub, min(16, self.n - 1))[:16]
            order = order[np.argsort(-ub[order], kind="stable")]
            vals = sorted(((-g, v) for v, g in got.items()))
            rest = ub[order[0]]
            if rest < 0 or (len(vals) >= need and rest * (1 + 1e-11) < -vals[need - 1][0]):
                return [(-g, v) for g, v in vals]
            cand = [int(v) for v in order if ub[v] >= 0]
            for v, g in zip(cand, self.columns(mask, phi, cand)):
                got[v] = float(g)
                stale[v] = min(stale[v], float(g))
                ub[v] = -1.0

    def sample(self, seed, step, k):
        m = math.ceil(self.n / k * math.log(1.0 / 0.1))
        p = m / (self.n - step)
        if p >= 1.0:
            return None
        with np.errstate(over="ignore"):
            z = np.uint64(seed) ^ np.uint64(step << 32) ^ np.arange(self.n, dtype=np.uint64)
            z = z + np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = z ^ (z >> np.uint64(31))
        return z < np.uint64(int(p * 2.0 ** 64))

    def maximize(self, k, eps, seed):
        L, _, B = self.length(eps / k)
        ell = 1 if self.case.get("adaptive") else L
        top = 1
        while top < L:
            top *= 2
        if self.case.get("adaptive"):
            _, _, B = self.length(B[L] * 1e-12) if top > L else (0, 0, B)
        S, gains, lengths = [], [], []
        stale = np.full(self.n, np.inf)
        for step in range(k):
            allowed = self.sample(seed, step, k) if self.case.get("stochastic") else None
            while True:
                vals = self.best(S, ell, 2 if self.case.get("adaptive") else 1, stale, allowed)
                if not self.case.get("adaptive") or vals[0][0] > vals[1][0] + B[ell] - eps / k:
                    break
                ell *= 2
                stale[:] = np.inf
            S.append(vals[0][1])
            gains.append(vals[0][0])
            lengths.append(ell)
        return S, np.array(gains), lengths, L


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        E = _Exact(case, seed)
        rp, _ = _graph(case, seed)
        words, x, alpha = _step_inputs(case, seed, rp)
        alpha = float(np.float32(alpha))  # the step's vectors and its factor are 32-bit
        S = _set(case, seed)
        s = alpha * (E.A @ x.double())
        inS = torch.from_numpy(S).long().cuda()
        y = s.clone()
        y[inS, 0] = s[inS].sum(1)
        y[inS, 1] = 0.0
        return {"y": y, "hit": y[:, 0].sum().reshape(1)}
    if kind in ("max", "fresh") and _nnz(case) * case["k"] > 1.8e9:
        return None
    E = _Exact(case, seed)
    if kind == "score":
        L, B, _ = E.length(case["eps"])
        return {"score": E.scores([_set(case, seed)], L)[0], "L": L, "bound": B}
    if kind == "batch":
        L, _, _ = E.length(case["eps"])
        off, mem = _groups(case, seed)
        return {"scores": E.scores([mem[off[j]:off[j + 1]] for j in range(len(off) - 1)], L), "L": L}
    if kind == "gains":
        L, _, _ = E.length(case["eps"])
        S = _set(case, seed)
        mask = E._mask(S)
        phi = E.table(mask, L, E.A)
        g = np.zeros(E.n)
        rest = np.setdiff1d(np.arange(E.n), S)
        for a in range(0, len(rest), 512):
            g[rest[a:a + 512]] = E.columns(mask, phi, rest[a:a + 512])
        return {"gains": g, "L": L}
    S, gains, lengths, L = E.maximize(case["k"], case["eps"], seed)
    score = E.scores([S], L)[0]
    out = {"group": None, "gains": gains, "score": score, "L": None}
    if case.get("adaptive"):
        out["lengths"] = None
    if kind == "fresh":
        out.update(nnz=None, dmax=None)
    return out
