"""The allocation-free step where a block makes several iterations over its rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [262_144, 262_145, 524_293, 800_011])  # 1, 2, 3 and 4 iterations of 32 rows a block
def test_rows_of_several_iterations(cuda_device, n):
    # sparse rows, hubs of each class (a warp's, a block's) at both ends and in the middle; the reference is
    # the same step in FP64, the tolerance that of the other allocation-free tests
    import torch

    from paper_1910_13874_gb300 import gedwalk

    rng = np.random.default_rng(n)
    deg = rng.integers(0, 7, size=n)
    for at, d in ((0, 5000), (1, 300), (n // 2, 2049), (n // 2 + 1, 257), (n - 1, 4097), (n - 2, 1000)):
        deg[at] = d
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    ci = rng.integers(0, n, size=int(rp[-1])).astype(np.int32)
    S = rng.choice(n, size=500, replace=False)
    words = np.zeros((n + 31) // 32, dtype=np.uint32)
    np.bitwise_or.at(words, S >> 5, np.uint32(1) << (S & 31).astype(np.uint32))
    x = rng.random((n, 2)).astype(np.float32)
    t = [torch.from_numpy(a).to(cuda_device) for a in (rp, ci, words.view(np.int32), x)]
    y = torch.full_like(t[3], -1.0)
    hit = torch.zeros(1, dtype=torch.float64, device=cuda_device)
    alpha = 2.0 ** -13
    gedwalk.score_step_noalloc(*[a.data_ptr() for a in t[:2]], n, t[2].data_ptr(), t[3].data_ptr(), y.data_ptr(), alpha,
                               hit.data_ptr(), torch.cuda.current_stream().cuda_stream)
    s = np.zeros((n, 2))
    np.add.at(s, np.repeat(np.arange(n), deg), x[ci].astype(np.float64))
    s *= alpha
    want = s.copy()
    want[S, 0] = s[S].sum(1)
    want[S, 1] = 0.0
    got = y.cpu().numpy().astype(np.float64)
    assert np.all(got[want == 0.0] == 0.0)
    assert np.max(np.abs(got - want) / np.maximum(want, 1e-30)) < 1e-5
    assert abs(hit.item() - want[:, 0].sum()) < 1e-6 * want[:, 0].sum()
