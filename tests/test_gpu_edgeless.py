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
