"""Graphs without edges: accepted by every call, all values 0, ties by lowest id."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 300])
@pytest.mark.parametrize("kind", ["plain", "weighted", "directed"])
def test_calls_on_an_edgeless_graph(cuda_device, n, kind):
    from paper_1910_13874_gb300 import gedwalk

    g = gg.from_edges(n, [])
    G = gedwalk.Graph.from_host(g, weighted=kind == "weighted", directed=kind == "directed")
    off, mem = np.array([0, 1, 1, 1 + n], dtype=np.int32), np.concatenate([[0], np.arange(n)]).astype(np.int32)
    for L in (1, 2, 13):
        scores, _ = G.score_batch(off, mem, L=L)
        assert np.array_equal(scores, np.zeros(3))
        for prec in ("fp64", "fp32"):
            assert G.score([0], precision=prec, L=L)[0] == 0.0
            assert np.array_equal(G.gains([0], precision=prec, L=L)[0], np.zeros(n))
            for kw in ({}, dict(gains_all=True), dict(stochastic=True)):
                grp, gains, score, _ = G.maximize(n, precision=prec, L=L, **kw)
                assert sorted(grp) == list(range(n)) and score == 0.0 and not np.any(gains)
                if "stochastic" not in kw:
                    assert list(grp) == list(range(n))
    G.free()


def test_serving_an_edgeless_graph(cuda_device):
    from paper_1910_13874_gb300 import gedwalk

    G = gedwalk.Graph.from_host(gg.from_edges(40, []))
    srv = gedwalk.Server([G])
    t = srv.submit_score(0, [1, 2])
    assert srv.poll(t, wait_us=30_000_000)["score"] == 0.0
    srv.close()
    G.free()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_zero_gains_in_the_sample_go_to_the_lowest_id(cuda_device, prec):
    # ten stars: once the centres are taken, bounds of 0 decide, in every block of the pass, and the lowest id
    # wins; in a sample, the leaves of an open star have equal gains (to rounding: the checker allows any of
    # them) and those of a taken one 0
    import oracle
    from seqcheck import check_sequence, oracle_stochastic_checker
    from paper_1910_13874_gb300 import gedwalk

    leaves, stars = 400, 10
    c = np.arange(stars) * (leaves + 1)
    e = np.concatenate([np.stack([np.full(leaves, x), x + 1 + np.arange(leaves)], 1) for x in c])
    g = gg.from_edges(stars * (leaves + 1), e)
    alpha = oracle.default_alpha(g)
    G = gedwalk.Graph.from_host(g)
    grp, gains, _, _ = G.maximize(16, precision=prec, L=6)
    assert sorted(grp[:10]) == list(c) and list(grp[10:]) == [1, 2, 3, 4, 5, 6] and not np.any(gains[10:])
    k, eta, tol = 60, 0.2, {"fp64": 1e-12, "fp32": 1e-5}[prec]
    grp, gains, _, _ = G.maximize(k, precision=prec, L=4, stochastic=True, eta=eta, seed=3)
    ref, ref_gains, _ = oracle.greedy_stochastic(g, k, alpha, 4, eta, 3)
    check_sequence(grp, gains, tol, ref, ref_gains, *oracle_stochastic_checker(oracle, g, alpha, 4, k, eta, 3))
    G.free()
