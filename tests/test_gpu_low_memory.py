"""Calls on a device that refuses large blocks: shorter rings, narrower rows, and at last two vectors.

The allocator hook returns NULL above a limit, set after the graph and its walk totals are there. Values
must stay within the tolerances of the calls without a limit: FP64 1e-12, FP32 1e-5 relative to the oracle.
"""
import contextlib
import functools

import numpy as np
import pytest

import graphgen as gg
import oracle
from seqcheck import check_sequence, oracle_greedy_checker, oracle_stochastic_checker

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 1e-5}


def rel(a, b):
    return abs(a - b) / max(abs(b), 1e-300)


@contextlib.contextmanager
def limited_allocator():
    """Yields a dict whose "limit" (bytes) larger requests fail above; "largest" is the largest block given
    since it was last reset."""
    import torch

    from paper_1910_13874_gb300 import gedwalk

    state = {"limit": None, "largest": 0, "live": {}}

    def alloc(nbytes, stream, ctx):
        if state["limit"] is not None and nbytes > state["limit"]:
            return None
        t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
        state["live"][t.data_ptr()] = t
        state["largest"] = max(state["largest"], int(nbytes))
        return t.data_ptr()

    def free(ptr, nbytes, stream, ctx):
        state["live"].pop(ptr, None)

    hooks = (gedwalk._ALLOC_FN(alloc), gedwalk._FREE_FN(free))
    gedwalk._hook_refs.append(hooks)  # blocks are freed through the hooks that made them
    assert gedwalk.load().gedwalk_set_allocator(hooks[0], hooks[1], None) == gedwalk.OK
    try:
        yield state
    finally:
        assert gedwalk.load().gedwalk_set_allocator(gedwalk._ALLOC_FN(), gedwalk._FREE_FN(), None) == gedwalk.OK
        gedwalk._torch_hooks = None
        gedwalk.use_torch_allocator()


@functools.lru_cache(maxsize=None)
def ba(n):
    return gg.barabasi_albert(n, 3, 4)


def upload(g, weighted=False, directed=False, longest=24):
    """The graph on the device with its walk totals to `longest`."""
    from paper_1910_13874_gb300 import gedwalk

    G = gedwalk.Graph.from_host(g, weighted=weighted, directed=directed)
    eps = 1e-3
    while G.truncation(epsilon=eps)[0] < longest:
        eps *= 1e-2
    w = oracle.normalized_weights(g) if weighted else None
    return G, w, oracle.default_alpha(g, w, directed)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("vectors", [5, 7, 2])  # a ring of three and its sum, of five, the two-state sweeps
def test_score_in_a_ring(cuda_device, prec, weighted, vectors):
    g = ba(8000)
    S = [0, 5, 699, 41]
    with limited_allocator() as state:
        G, w, alpha = upload(g, weighted)
        state.update(limit=vectors * g.n * 2 * (8 if prec == "fp64" else 4), largest=0)
        for L in (3, 7, 12, 13, 18, 19, 23, 24):
            for _ in range(3):  # direct and captured
                got, _, _ = G.score(S, precision=prec, L=L)
            assert rel(got, oracle.score(g, S, alpha, L, w=w)) < TOL[prec], L
        assert state["largest"] <= state["limit"]
        state["limit"] = None
        G.free()


@pytest.mark.parametrize("width", [8, 32])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("cols", [0, 4, 8])  # a ring of two at the width set, or blocks of so many columns
def test_batch_in_little_memory(cuda_device, width, weighted, cols):
    g = ba(3000)
    off, mem = gg.random_groups(g.n, width + 3, 0, 9, 3)
    with limited_allocator() as state:
        G, w, alpha = upload(g, weighted)
        G.batch_set_width(width)
        state.update(limit=4 * g.n * 4 * (cols or width), largest=0)
        for L in (1, 5, 6, 9, 10, 11, 14, 23):
            scores, _ = G.score_batch(off, mem, L=L)
            for j in (0, 1, width - 1, width, width + 2):
                S = mem[off[j]:off[j + 1]]
                want = oracle.score(g, S, alpha, L, w=w)
                assert scores[j] == want == 0.0 or rel(scores[j], want) < 1e-5, (L, j)
        assert state["largest"] <= state["limit"]
        state["limit"] = None
        G.free()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["plain", "weighted", "directed", "stochastic", "gains_all"])
@pytest.mark.parametrize("cols", [4, 2])
def test_greedy_on_narrow_rows(cuda_device, prec, kind, cols):
    from paper_1910_13874_gb300 import gedwalk

    directed = kind == "directed"
    g = gg.rmat(13, 8, seed=6, directed=True) if directed else ba(14_000 if kind == "gains_all" else 8192)
    k, L = {"gains_all": 1, "stochastic": 2}.get(kind, 9), 13
    with limited_allocator() as state:
        G, w, alpha = upload(g, kind == "weighted", directed)
        if directed:
            G.batch_set_width(8)  # the tuner would leave large blocks behind
            srv = gedwalk.Server([G])  # a submitted request makes the second table of walk totals
            srv.poll(srv.submit_maximize(0, 1, L=L))
            srv.close()
        H, sets = (L + 1) // 2, 2 if directed else 1
        vec = g.n * H * sets * (8 if prec == "fp64" else 4)
        state.update(limit=vec * cols + 8 * g.n * (sets if kind == "weighted" else 1) * cols, largest=0)
        kw = dict(stochastic=True, eta=0.3, seed=5) if kind == "stochastic" else dict(gains_all=True) if kind == "gains_all" else {}
        gedwalk.profile(True)
        grp, gains, score, _ = G.maximize(k, precision=prec, L=L, **kw)
        top = gedwalk.profile_read()["top_cols"]
        gedwalk.profile(False)
        assert top <= cols and state["largest"] <= state["limit"]
        state["limit"] = None
        G.free()
    if kind == "stochastic":
        ref, ref_gains, _ = oracle.greedy_stochastic(g, k, alpha, L, 0.3, 5)
        check = oracle_stochastic_checker(oracle, g, alpha, L, k, 0.3, 5)
    else:
        ref, ref_gains, _ = oracle.greedy(g, k, alpha, L, "lazy", w=w, directed=directed)
        check = oracle_greedy_checker(oracle, g, alpha, L, w=w, directed=directed)
    check_sequence(grp, gains, TOL[prec], ref, ref_gains, *check)


def test_gains_on_narrow_rows(cuda_device):
    g = ba(14_000)
    with limited_allocator() as state:
        G, _, alpha = upload(g)
        state.update(limit=8 * g.n * 7 * 4, largest=0)
        gains, _ = G.gains([3, 44], precision="fp32", L=13)
        assert state["largest"] <= state["limit"]
        state["limit"] = None
        for x in (0, 17, 6000, 13_999):
            assert rel(gains[x], oracle.gain(g, [3, 44], x, alpha, 13)) < 1e-5, x
        G.free()


def test_served_directed_requests_run_narrower_in_a_small_budget(cuda_device):
    from paper_1910_13874_gb300 import gedwalk

    g = gg.rmat(13, 8, seed=6, directed=True)
    G = gedwalk.Graph.from_host(g, directed=True)
    srv = gedwalk.Server([G], mem_budget=1 << 34)
    alone = srv.poll(srv.submit_maximize(0, 30))
    F = srv.stats()["peak_bytes"]
    srv.close()
    budget = int(1.8 * F)
    srv = gedwalk.Server([G], mem_budget=budget)
    res = [srv.poll(t) for t in [srv.submit_maximize(0, 30) for _ in range(4)]]
    st = srv.stats()
    srv.close()
    G.free()
    assert st["peak_maximize_running"] >= 2 and st["peak_bytes"] <= budget, st
    for r in res:
        assert list(r["group"]) == list(alone["group"])
        assert np.allclose(r["gains"], alone["gains"], rtol=1e-6, atol=0)
