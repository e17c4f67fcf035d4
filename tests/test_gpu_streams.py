"""Calls on every kind of stream handle, often enough that their launch sequences are captured and replayed."""
import numpy as np
import pytest

import graphgen as gg
import oracle

pytestmark = pytest.mark.gpu

LEGACY, PER_THREAD = 1, 2  # cudaStreamLegacy, cudaStreamPerThread


@pytest.mark.parametrize("handle", [0, LEGACY, PER_THREAD, None])
@pytest.mark.parametrize("directed", [False, True])
def test_repeated_calls(cuda_device, handle, directed):
    import torch

    from paper_1910_13874_gb300 import gedwalk

    stream = torch.cuda.Stream()
    h = stream.cuda_stream if handle is None else handle
    g = gg.rmat(9, 8, seed=6, directed=directed)
    alpha = oracle.default_alpha(g, directed=directed)
    G = gedwalk.Graph.from_host(g, directed=directed)
    S, L = [1, 2, 40], 5
    want = oracle.score(g, S, alpha, L)
    ref, _, _ = oracle.greedy(g, 4, alpha, L, "lazy", directed=directed)
    off, mem = np.array([0, 3], dtype=np.int32), np.array(S, dtype=np.int32)
    for _ in range(4):
        assert abs(G.score(S, precision="fp64", L=L, stream=h)[0] - want) <= 1e-12 * want
        assert abs(G.score_batch(off, mem, L=L, stream=h)[0][0] - want) <= 1e-5 * want
        assert list(G.maximize(4, precision="fp64", L=L, stream=h)[0]) == list(ref)
        gain = G.gains(S, precision="fp64", L=L, stream=h)[0][7]
        ref_gain = oracle.gain(g, S, 7, alpha, L)
        assert abs(gain - ref_gain) <= 1e-12 * ref_gain
    G.free()
