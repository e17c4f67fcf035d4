"""The half-length runs at the sizes where their pieces change over, against the CPU oracle.

Odd and even walk lengths from 1 on, a batch long enough to fold its ring of vectors at every column
width, the gains in shared memory on both sides of each column count, row lengths on both sides of
every network of the upload's row sort, the allocation-free step's row classes, and chains of both
FP64 widths. Tolerances as for the other parity tests: FP64 1e-12, FP32 1e-5 relative.
"""
import functools

import numpy as np
import pytest

import graphgen as gg
import oracle
from seqcheck import check_sequence, oracle_greedy_checker

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5}


def rel(a, b):
    return abs(a - b) / max(abs(b), 1e-300)


@functools.lru_cache(maxsize=None)
def ba():
    return gg.barabasi_albert(700, 3, 4)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("weighted", [False, True])
def test_lengths(cuda_device, prec, weighted):
    from paper_1910_13874_gb300 import gedwalk

    g = ba()
    w = oracle.normalized_weights(g) if weighted else None
    alpha = oracle.default_alpha(g, w)
    G = gedwalk.Graph.from_host(g, weighted=weighted)
    S = [0, 5, 699, 41]
    for L in (1, 2, 3, 4, 5, 8, 11):
        got, _, _ = G.score(S, precision=prec, alpha=alpha, L=L)
        assert rel(got, oracle.score(g, S, alpha, L, w=w)) < TOL[prec], L
        grp, gains, _, _ = G.maximize(4, precision=prec, alpha=alpha, L=L)
        ref, ref_gains, _ = oracle.greedy(g, 4, alpha, L, "lazy", w=w)
        check_sequence(grp, gains, TOL[prec], ref, ref_gains, *oracle_greedy_checker(oracle, g, alpha, L, w=w))
    G.free()


@pytest.mark.parametrize("width", [8, 16, 32, 64])
@pytest.mark.parametrize("weighted", [False, True])
def test_batch_folds_long_walks(cuda_device, width, weighted):
    from paper_1910_13874_gb300 import gedwalk

    g = ba()
    w = oracle.normalized_weights(g) if weighted else None
    alpha = oracle.default_alpha(g, w)
    G = gedwalk.Graph.from_host(g, weighted=weighted)
    G.batch_set_width(width)
    off, mem = gg.random_groups(g.n, width + 3, 0, 9, 3)
    for L in (1, 2, 9, 10, 11, 12, 19, 20, 27):  # H = 5 fills the ring, 6, 10 and 14 fold it
        scores, _ = G.score_batch(off, mem, alpha=alpha, L=L)
        for j in (0, 1, width - 1, width, width + 2):
            S = mem[off[j]:off[j + 1]]
            want = oracle.score(g, S, alpha, L, w=w)
            assert scores[j] == want == 0.0 or rel(scores[j], want) < 1e-5, (L, j)
    G.free()


@pytest.mark.parametrize("prec,n", [("fp32", 3200), ("fp32", 3201), ("fp32", 6401), ("fp32", 12801), ("fp64", 1600),
                                    ("fp64", 1601), ("fp64", 3201), ("fp64", 6401)])
def test_gains_at_the_column_counts(cuda_device, prec, n):
    # 200 KiB hold 8, 4 or 2 columns of two vectors up to these sizes; beyond, candidate runs
    from paper_1910_13874_gb300 import gedwalk

    g = gg.erdos_renyi(n, 30, 2)  # no isolated vertex; rows on both sides of 64 after the hub below
    hub = [(0, v) for v in range(1, 200)]
    rows = np.repeat(np.arange(n), np.diff(g.row_ptr))
    g = gg.from_edges(n, np.concatenate([np.stack([rows, g.col_idx], 1), hub]))
    alpha = oracle.default_alpha(g)
    G = gedwalk.Graph.from_host(g)
    S, L = [3, 17], 3
    gains, _ = G.gains(S, precision=prec, L=L)
    assert gains[3] == gains[17] == 0.0
    for x in (0, 1, 2, 4, n // 2, n - 2, n - 1):
        assert rel(gains[x], oracle.gain(g, S, x, alpha, L)) < TOL[prec], x
    G.free()


def test_rows_at_the_sort_networks(cuda_device):
    # one vertex of every length around a network's size, joined to a common pool in shuffled order
    from paper_1910_13874_gb300 import gedwalk

    sizes = [1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 256, 257, 512, 513, 1024, 1025, 2049]
    rng = np.random.default_rng(1)
    pool = np.arange(len(sizes), len(sizes) + 2200)
    edges = [(i, int(v)) for i, d in enumerate(sizes) for v in rng.choice(pool, size=d, replace=False)]
    g = gg.from_edges(len(sizes) + 2200, edges)
    alpha = oracle.default_alpha(g)
    G = gedwalk.Graph.from_host(g)
    for i in range(len(sizes)):
        got, _, _ = G.score([i], precision="fp64", L=4)
        assert rel(got, oracle.score(g, [i], alpha, 4)) < 1e-12, sizes[i]
    G.free()


def test_noalloc_row_classes(cuda_device):
    # rows of 0 to 32, 33 to 256, 257 to 2048 and above 2048 entries, and a row count that is no
    # multiple of a block's; the reference is the same step in FP64
    import torch

    from paper_1910_13874_gb300 import gedwalk

    rng = np.random.default_rng(2)
    n = 5003
    deg = rng.integers(0, 40, size=n)
    deg[:8] = [255, 256, 257, 2047, 2048, 2049, 4096, 4999]
    deg[4990:4994] = [300, 2500, 31, 32]
    rows = [np.sort(rng.choice(n, size=int(d), replace=False)) for d in deg]
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    ci = np.concatenate(rows).astype(np.int32)
    S = rng.choice(n, size=60, replace=False)
    words = np.zeros((n + 31) // 32, dtype=np.uint32)
    np.bitwise_or.at(words, S >> 5, np.uint32(1) << (S & 31).astype(np.uint32))
    x = rng.random((n, 2)).astype(np.float32)
    t = [torch.from_numpy(a).to(cuda_device) for a in (rp, ci, words.view(np.int32), x)]
    y = torch.empty_like(t[3])
    hit = torch.zeros(1, dtype=torch.float64, device=cuda_device)
    alpha = 1.0 / 5000
    gedwalk.score_step_noalloc(*[a.data_ptr() for a in t[:2]], n, t[2].data_ptr(), t[3].data_ptr(), y.data_ptr(), alpha,
                               hit.data_ptr(), torch.cuda.current_stream().cuda_stream)
    s = np.array([x[r].astype(np.float64).sum(0) for r in rows]) * float(np.float32(alpha))
    want = s.copy()
    want[S, 0] = s[S].sum(1)
    want[S, 1] = 0.0
    got = y.cpu().numpy().astype(np.float64)
    assert np.all(got[want == 0.0] == 0.0)
    assert np.max(np.abs(got - want) / np.maximum(want, 1e-30)) < 1e-5
    assert rel(hit.item(), want[:, 0].sum()) < 1e-6


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("L", [1, 2, 5, 6])
def test_directed_lengths(cuda_device, prec, L):
    from paper_1910_13874_gb300 import gedwalk

    g = gg.rmat(9, 8, seed=6, directed=True)
    alpha = oracle.default_alpha(g, directed=True)
    G = gedwalk.Graph.from_host(g, directed=True)
    grp, gains, score, _ = G.maximize(10, precision=prec, L=L)
    ref, ref_gains, _ = oracle.greedy(g, 10, alpha, L, "lazy", directed=True)
    check_sequence(grp, gains, TOL[prec], ref, ref_gains, *oracle_greedy_checker(oracle, g, alpha, L, directed=True))
    assert rel(score, oracle.score(g, grp, alpha, L)) < TOL[prec]
    every, _ = G.gains(grp[:3], precision=prec, L=L)
    for x in np.random.default_rng(3).choice(g.n, 20, replace=False):
        want = oracle.gain(g, grp[:3], int(x), alpha, L)
        assert every[x] == want == 0.0 or rel(every[x], want) < TOL[prec], x
    G.free()


def test_fp64_chain_widths(cuda_device):
    # above 20,000 vertices an FP64 maximisation starts with chains of seven steps, below with three,
    # and widens once a chain held: both against the oracle
    from paper_1910_13874_gb300 import gedwalk

    for n in (3000, 30_000):
        g = gg.barabasi_albert(n, 4, 8)
        alpha = oracle.default_alpha(g)
        G = gedwalk.Graph.from_host(g)
        grp, gains, _, L = G.maximize(16, precision="fp64", epsilon=1e-2)
        ref, ref_gains, _ = oracle.greedy(g, 16, alpha, L, "lazy")
        check_sequence(grp, gains, 1e-12, ref, ref_gains, *oracle_greedy_checker(oracle, g, alpha, L))
        G.free()


@pytest.mark.parametrize("kw", [{}, dict(lookahead=1)])
def test_long_walks_are_certified(cuda_device, kw):
    # 30 sweeps a run: the rounding a certification allows for grows with the root of their number
    from paper_1910_13874_gb300 import gedwalk

    g = gg.erdos_renyi(2000, 8, 5)
    alpha = oracle.default_alpha(g)
    G = gedwalk.Graph.from_host(g)
    grp, gains, _, _ = G.maximize(12, precision="fp32", L=61, **kw)
    ref, ref_gains, _ = oracle.greedy(g, 12, alpha, 61, "lazy")
    check_sequence(grp, gains, 1e-5, ref, ref_gains, *oracle_greedy_checker(oracle, g, alpha, 61))
    G.free()


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("size", [1, 7, 9, 2000])
def test_groups_of_every_size(cuda_device, directed, size):
    # one warp per member and more slices for the rows above 256 entries: a hub of 2500, groups with and
    # without it, up to half of the graph, scored and as an init group
    from paper_1910_13874_gb300 import gedwalk

    n = 4000
    rng = np.random.default_rng(size)
    arcs = np.concatenate([rng.integers(0, n, size=(8 * n, 2)), [(0, v) for v in range(1, 2501)], [(v, 1) for v in range(2, 1500)]])
    g = gg.from_arcs(n, arcs) if directed else gg.from_edges(n, arcs)
    alpha = oracle.default_alpha(g, directed=directed)
    G = gedwalk.Graph.from_host(g, directed=directed)
    rest = rng.permutation(np.arange(2, n))
    for S in (rest[:size], np.concatenate([[0, 1], rest[:size]])):
        for _ in range(3):  # direct and captured
            got, _, _ = G.score(S, precision="fp64", L=5)
        assert rel(got, oracle.score(g, S, alpha, 5)) < 1e-12
        _, gains, score, _ = G.maximize(1, precision="fp64", L=5, init=S)
        _, ref_gains, _ = oracle.greedy(g, 1, alpha, 5, "lazy", init=list(S), directed=directed)
        assert rel(gains[0], ref_gains[0]) < 1e-12
        assert rel(score, oracle.score(g, S, alpha, 5) + ref_gains[0]) < 1e-12
    G.free()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["plain", "weighted", "directed"])
def test_alpha_beyond_the_bound(cuda_device, prec, kind):
    # a forced length with alpha * d_max > 1: no table of walk totals applies, the call makes its own
    from paper_1910_13874_gb300 import gedwalk

    directed = kind == "directed"
    g = gg.rmat(9, 8, seed=6, directed=True) if directed else ba()
    w = oracle.normalized_weights(g) if kind == "weighted" else None
    alpha = 2.5 / oracle.delta(g, w, directed)
    G = gedwalk.Graph.from_host(g, weighted=kind == "weighted", directed=directed)
    for L in (1, 2, 3, 8, 11):
        for init in (None, [3, 17, 200]):
            grp, gains, _, _ = G.maximize(6, precision=prec, alpha=alpha, L=L, init=init)
            ref, ref_gains, _ = oracle.greedy(g, 6, alpha, L, "lazy", init=init, w=w, directed=directed)
            if init is None:
                check_sequence(grp, gains, TOL[prec], ref, ref_gains,
                               *oracle_greedy_checker(oracle, g, alpha, L, w=w, directed=directed))
            else:
                assert np.allclose(gains, ref_gains, rtol=TOL[prec], atol=0), L
    G.free()


def test_sweeps_are_counted_for_gains_from_shared_memory(cuda_device):
    from paper_1910_13874_gb300 import gedwalk

    G = gedwalk.Graph.from_host(ba())
    G.maximize(3, precision="fp32", L=7, gains_all=True)
    assert G.maximize_stats()["sweeps"] == 3 * 4  # phi^miss to half the length, per step
    G.free()
