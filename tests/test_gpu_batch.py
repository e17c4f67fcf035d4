"""Batched scoring where its parts are at their limits, against the CPU oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu


def rel(a, b):
    return abs(a - b) / max(abs(b), 1e-300)


def star(leaves):
    e = np.stack([np.zeros(leaves, dtype=np.int64), np.arange(1, leaves + 1)], 1)
    return gg.from_edges(leaves + 1, e)


@pytest.mark.parametrize("leaves", [2000, 10_000, 100_000])
def test_many_members_at_one_vertex(cuda_device, leaves):
    # h_1 of the centre counts half of the leaves. A count times alpha is rounded once and the walks of
    # length 6 pass a handful of roundings of 6e-8 each, so 1e-6 holds; adding alpha up 50,000 times is off
    # by 2.7e-4.
    from paper_1910_13874_gb300 import gedwalk

    g = star(leaves)
    alpha = oracle.default_alpha(g)
    rng = np.random.default_rng(leaves)
    groups = [1 + rng.choice(leaves, leaves // 2, replace=False), [0], [1, 2, 3], np.arange(1, leaves + 1)]
    off = np.concatenate([[0], np.cumsum([len(S) for S in groups])]).astype(np.int32)
    mem = np.concatenate(groups).astype(np.int32)
    G = gedwalk.Graph.from_host(g)
    for L in (1, 2, 6):
        scores, _ = G.score_batch(off, mem, alpha=alpha, L=L)
        for j, S in enumerate(groups):
            assert rel(scores[j], oracle.score(g, S, alpha, L)) < 1e-6, (L, j)
    G.free()
