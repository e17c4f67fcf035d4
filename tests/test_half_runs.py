"""The identities behind the runs of half the walk length, against walk-by-walk recurrences on the CPU.

A walk of length a + b that avoids S is two such walks, of lengths a and b, that end at the same
vertex, so the walks through a candidate number <k_a, phi_b> + <phi_a - k_a, k_b>; and with first
visits bounded through the immediate returns the bound of a vertex is F + U + F U plus the pairs
longer than the stored half, taken from the empty set.
"""
import numpy as np
import pytest

import graphgen as gg


def graphs():
    return {"er": gg.random_graph_small(40, 0.12, 3), "star": gg.star(12), "path": gg.path(15), "k6": gg.complete(6),
            "ba": gg.barabasi_albert(60, 3, 5),
            "parts": gg.from_edges(12, [(0, 1), (1, 2), (2, 0), (4, 5), (6, 7), (7, 8)])}


def table(M, L, x0):
    rows = [x0]
    for _ in range(L):
        rows.append(M @ rows[-1])
    return np.array(rows)


def column(M, phi, c, base):
    """Walks through c that avoid `base`: k_0 = e_c, k_t = M k_{t-1}, k_t(c) = phi_t(c)."""
    k = np.zeros_like(phi)
    k[0, c] = 1.0
    for t in range(1, len(phi)):
        k[t] = M @ k[t - 1]
        k[t, c] = phi[t, c]
    return k


@pytest.mark.parametrize("name", list(graphs()))
@pytest.mark.parametrize("L", [1, 2, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("weighted", [False, True])
def test_half_length_gain_and_bound(name, L, weighted):
    g = graphs()[name]
    A = g.to_dense().astype(float)
    if weighted:
        s = np.random.default_rng(5).uniform(0.2, 1.0, g.n)
        A = A * s[:, None] * s[None, :]
    alpha = 1.0 / (1.0 + A.sum(1).max())
    S = [1, 4]
    mask = np.ones(g.n)
    mask[S] = 0.0
    M = alpha * mask[:, None] * A
    H = (L + 1) // 2
    phi = table(M, L, mask)
    full = table(alpha * A, L, np.ones(g.n))
    Qf = full.cumsum(0)
    tail = 2 * sum((full[a] * Qf[L - a] for a in range(H + 1, L + 1)), np.zeros(g.n))
    deg = (A > 0) @ mask
    for c in range(g.n):
        if c in S:
            continue
        k = column(M, phi, c, S)
        want = k[1:].sum()
        V = k[1:L - H + 1].sum(0)
        P = phi[1:L - H + 1].sum(0)
        got = (k[1:H + 1].sum(0) + V * phi[H] + (P - V) * k[H]).sum()
        assert got == pytest.approx(want, rel=1e-12, abs=1e-15)
        # the bound: first visits less the closed walks c-u-c and c-u-v-u-c
        U = phi[1:H + 1, c].sum()
        if deg[c] == 0:
            assert want == 0.0
            continue
        if weighted:
            s2, s4 = phi[1, c] ** 2 / deg[c], 0.0
        else:
            s2 = alpha ** 2 * deg[c]
            s4 = max(0.0, alpha ** 2 * (phi[2, c] if L >= 2 else 0.0) - alpha ** 3 * phi[1, c])
        corr = 0.0
        if H >= 2:
            corr += s2 * (1 + phi[1:H - 1, c].sum())
        if H >= 4:
            corr += s4 * (1 + phi[1:H - 3, c].sum())
        F = U - corr
        ub = F + U + F * U + tail[c]
        if L % 2:
            ub -= phi[H, c] * max(0.0, phi[H, c] - corr)
        assert ub >= want * (1 - 1e-12)
        # never above the bound that pairs all visits with all continuations, but for the tail
        Q = phi.cumsum(0)
        lemma = sum(phi[a, c] * Q[L - a, c] for a in range(1, L + 1)) + (Q[L, c] - phi[0, c])
        assert ub <= lemma + tail[c] + phi[H, c] * corr + 1e-12


@pytest.mark.parametrize("name", ["er", "ba", "k6"])
def test_half_length_chain(name):
    # candidate j of a chain runs under S + the earlier candidates; its level's phi is column 0 less
    # the columns before it
    g = graphs()[name]
    A = g.to_dense().astype(float)
    alpha = 1.0 / (1.0 + A.sum(1).max())
    L, H = 7, 4
    S, chain = [0], [3, 5, 1]
    mask = np.ones(g.n)
    mask[S] = 0.0
    phi = table(alpha * mask[:, None] * A, L, mask)
    base = phi.copy()
    for c in chain:
        M = alpha * mask[:, None] * A
        assert np.allclose(base, table(M, L, mask), atol=1e-14)
        k = column(M, base, c, S)
        V, P = k[1:L - H + 1].sum(0), base[1:L - H + 1].sum(0)
        got = (k[1:H + 1].sum(0) + V * base[H] + (P - V) * k[H]).sum()
        assert got == pytest.approx(k[1:].sum(), rel=1e-12)
        base = base - k
        mask = mask.copy()
        mask[c] = 0.0


@pytest.mark.parametrize("L", [1, 2, 5, 6, 9])
def test_half_length_directed(L):
    # walks that start at a vertex along the rows, walks that end there along the reverse lists
    A = gg.random_digraph(40, 0.08, 7).to_dense().astype(float)
    alpha = 1.0 / (1.0 + A.sum(1).max())
    S, H = [1, 4], (L + 1) // 2
    mask = np.ones(40)
    mask[S] = 0.0
    Ma, Mb = alpha * mask[:, None] * A, alpha * mask[:, None] * A.T
    phi, psi = table(Ma, L, mask), table(Mb, L, mask)
    fa, fb = table(alpha * A, L, np.ones(40)), table(alpha * A.T, L, np.ones(40))
    Qa, Qb = fa.cumsum(0), fb.cumsum(0)
    tail = sum((fb[p] * Qa[L - p] + fa[p] * Qb[L - p] for p in range(H + 1, L + 1)), np.zeros(40))
    for c in range(40):
        if c in S:
            continue
        k, j = column(Ma, phi, c, S), column(Mb, psi, c, S)
        V, P = j[1:L - H + 1].sum(0), psi[1:L - H + 1].sum(0)
        got = (k[1:H + 1].sum(0) + V * phi[H] + (P - V) * k[H]).sum()
        assert got == pytest.approx(k[1:].sum(), rel=1e-12, abs=1e-15)
        U, F = phi[1:H + 1, c].sum(), psi[1:H + 1, c].sum()
        ub = F + U + F * U + tail[c] - (phi[H, c] * psi[H, c] if L % 2 else 0.0)
        assert ub >= k[1:].sum() * (1 - 1e-12)
