"""FP32 calls on graphs whose walk vectors FP32 holds exactly, against the CPU oracle.

With alpha a power of two (and vertex scales 1 or 2) a stored walk vector is a whole number below 2^24 times
a power of two, so sweeps do not round. What is left are the sums over walk lengths and vertices and the
products in which half walks meet. Those are kept as pairs of FP32 values or in FP64 and are good to 2^-46:
1e-12 after some hundreds of additions, where one FP32 rounding would show as 1e-8.
"""
import functools

import numpy as np
import pytest

import graphgen as gg
import oracle
from seqcheck import check_sequence, oracle_greedy_checker

pytestmark = pytest.mark.gpu

ALPHA = 2.0 ** -10
TOL = 1e-12


def rel(a, b):
    return abs(a - b) / max(abs(b), 1e-300)


@functools.lru_cache(maxsize=None)
def ba(n):
    return gg.barabasi_albert(n, 3, 4)


def scales(g):
    return np.random.default_rng(g.n).integers(1, 3, size=g.n).astype(np.float64)


def upload(g, weighted):
    from paper_1910_13874_gb300 import gedwalk

    if not weighted:
        return gedwalk.Graph.from_host(g), None
    s = scales(g)
    return gedwalk.Graph.from_host(g, vertex_scale=s), np.repeat(s, np.diff(g.row_ptr)) * s[g.col_idx]


def check_greedy(G, g, k, L, w=None, directed=False, **kw):
    grp, gains, score, _ = G.maximize(k, precision="fp32", alpha=ALPHA, L=L, **kw)
    ref, ref_gains, _ = oracle.greedy(g, k, ALPHA, L, "lazy", w=w, directed=directed)
    check_sequence(grp, gains, TOL, ref, ref_gains, *oracle_greedy_checker(oracle, g, ALPHA, L, w=w, directed=directed))
    assert rel(score, sum(ref_gains)) < TOL


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("kw", [{}, dict(lookahead=3), dict(lookahead=1), dict(lookahead=1, spec_cols=8)])
def test_greedy_gains(cuda_device, weighted, kw):
    g = ba(700)
    G, w = upload(g, weighted)
    for L in (1, 2, 3, 5, 6):
        check_greedy(G, g, 9, L, w=w, **kw)
    G.free()


def test_directed_greedy_gains(cuda_device):
    from paper_1910_13874_gb300 import gedwalk

    g = gg.rmat(9, 8, seed=6, directed=True)
    G = gedwalk.Graph.from_host(g, directed=True)
    for L in (1, 2, 5, 6):
        check_greedy(G, g, 9, L, directed=True)
        check_greedy(G, g, 4, L, directed=True, spec_cols=4)
    S = [3, 44, 101]
    gains, _ = G.gains(S, precision="fp32", alpha=ALPHA, L=5)
    for x in range(0, g.n, 37):
        want = oracle.gain(g, S, x, ALPHA, 5)
        assert gains[x] == want == 0.0 or rel(gains[x], want) < TOL, x
    G.free()


@pytest.mark.parametrize("weighted", [False, True])
def test_gains_by_candidate_runs(cuda_device, weighted):
    g = ba(13_000)  # beyond the graphs whose gains come from shared memory
    G, w = upload(g, weighted)
    S = [3, 44, 12_000]
    for L in (2, 5):
        gains, _ = G.gains(S, precision="fp32", alpha=ALPHA, L=L)
        for x in (0, 1, 17, 600, 6000, 12_999):
            assert rel(gains[x], oracle.gain(g, S, x, ALPHA, L, w=w)) < TOL, (L, x)
    G.free()


@pytest.mark.parametrize("weighted", [False, True])
def test_score(cuda_device, weighted):
    g = ba(700)
    G, w = upload(g, weighted)
    for L in (1, 2, 3, 4, 5, 6, 7, 8):
        if weighted and L > 6:
            continue
        for S in ([0], [5, 699, 41], list(range(0, 700, 3))):
            got, _, _ = G.score(S, precision="fp32", alpha=ALPHA, L=L)
            assert rel(got, oracle.score(g, S, ALPHA, L, w=w)) < TOL, (L, len(S))
    G.free()


@pytest.mark.parametrize("n", [700, 5000, 9000])  # 8, 4 and 2 columns a block
@pytest.mark.parametrize("weighted", [False, True])
def test_gains_from_shared_memory(cuda_device, n, weighted):
    g = ba(n)
    G, w = upload(g, weighted)
    S = [3, 44, 611]
    for L in (1, 2, 3, 4, 5, 6):
        gains, _ = G.gains(S, precision="fp32", alpha=ALPHA, L=L)
        for x in (0, 1, 17, 600, n - 1):
            assert rel(gains[x], oracle.gain(g, S, x, ALPHA, L, w=w)) < TOL, (L, x)
    G.free()


def test_row_sums_of_the_small_gains(cuda_device):
    # 500 vertices joined to the same 63: most of a gain is sums of 63 equal terms, of a value whose running
    # FP32 sum drifts by 16 units in the last place (6e-7 of the gain). As a tree a sum takes six additions
    # of half a unit each, on both factors at most: 7 units, 4.2e-7.
    from paper_1910_13874_gb300 import gedwalk

    m, mids = 500, 63
    a, b = np.meshgrid(np.arange(m), m + np.arange(mids), indexing="ij")
    g = gg.from_edges(m + mids, np.stack([a.ravel(), b.ravel()], 1))
    alpha = float.fromhex("0x1.f08ccp+0")
    G = gedwalk.Graph.from_host(g)
    gains, _ = G.gains([], precision="fp32", alpha=alpha, L=4)
    for x in (0, 250, 499, m, m + 62):
        assert rel(gains[x], oracle.gain(g, [], x, alpha, 4)) < 4.2e-7, x
    G.free()


def test_hub_row_of_many_slices(cuda_device):
    # a hub's row is summed in slices of 1024 entries, here 488 equal ones. alpha has 19 bits, so a slice is
    # exact, and its multiples round the same way in a running sum: 7e-6 of the score. Compensated, a
    # handful of roundings of 6e-8 are left: 1e-6.
    from paper_1910_13874_gb300 import gedwalk

    g = gg.star(488 * 1024)
    alpha = 0x40007 * 2.0 ** -22
    want = oracle.score(g, [1], alpha, 6)
    G = gedwalk.Graph.from_host(g)
    assert rel(G.score([1], precision="fp32", alpha=alpha, L=6)[0], want) < 1e-6
    for width in (8, 64):
        G.batch_set_width(width)
        scores, _ = G.score_batch([0, 1, 2], [1, 7], alpha=alpha, L=6)
        assert rel(scores[0], want) < 1e-6 and rel(scores[1], want) < 1e-6
    G.free()
