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


def power_of_two_case(n, seed):
    """A graph of degree at most 3 with alpha = 2^-8 and vertex scales 1 or 2: every walk vector up to
    length 14 (6 with the scales) is a whole number below 2^24 times a power of two, so FP32 holds it exactly."""
    rng = np.random.default_rng(seed)
    ring = np.stack([np.arange(n), (np.arange(n) + 1) % n], 1)
    match = rng.permutation(n)[:n // 2 * 2].reshape(-1, 2)
    return gg.from_edges(n, np.concatenate([ring, match])), 2.0 ** -8, rng.integers(1, 3, size=n).astype(np.float64)


@pytest.mark.parametrize("width", [8, 16, 32, 64])
@pytest.mark.parametrize("weighted", [False, True])
def test_nothing_but_the_stored_vectors_is_fp32(cuda_device, width, weighted):
    # exact vectors leave the totals, products and sums: pairs of FP32 values carry 2^-46, some tens of
    # additions in a row stay below 1e-12 (one FP32 rounding would show as 1e-8)
    from paper_1910_13874_gb300 import gedwalk

    g, alpha, s = power_of_two_case(502, width)
    scale = s if weighted else None
    w = np.repeat(s, np.diff(g.row_ptr)) * s[g.col_idx] if weighted else None
    G = gedwalk.Graph.from_host(g, vertex_scale=scale)
    G.batch_set_width(width)
    off, mem = gg.random_groups(g.n, width + 3, 0, 9, 3)
    for L in (1, 2, 5, 9, 10, 12, 19, 27):
        if weighted and L > 12:
            continue  # the scales add up to two bits a step
        scores, _ = G.score_batch(off, mem, alpha=alpha, L=L)
        for j in (0, 1, width - 1, width, width + 2):
            S = mem[off[j]:off[j + 1]]
            want = oracle.score(g, S, alpha, L, w=w)
            assert scores[j] == want == 0.0 or rel(scores[j], want) < 1e-12, (L, j)
    G.free()
