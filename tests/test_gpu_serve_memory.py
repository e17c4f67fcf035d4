"""Served maximisations allocate no more than they are charged for, counted by an allocator hook."""
import threading

import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


def counting_allocator(state):
    """A PyTorch-backed allocator that adds up the live bytes of the other threads' allocations."""
    import torch

    from paper_1910_13874_gb300 import gedwalk

    me = threading.get_ident()

    def alloc(nbytes, stream, ctx):
        t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
        mine = threading.get_ident() == me
        state["blocks"][t.data_ptr()] = (t, 0 if mine else int(nbytes))
        if not mine:
            state["now"] += int(nbytes)
            state["peak"] = max(state["peak"], state["now"])
        return t.data_ptr()

    def free(ptr, nbytes, stream, ctx):
        state["now"] -= state["blocks"].pop(ptr)[1]

    hooks = (gedwalk._ALLOC_FN(alloc), gedwalk._FREE_FN(free))
    gedwalk._hook_refs.append(hooks)  # blocks are freed through the hooks that made them
    assert gedwalk.load().gedwalk_set_allocator(hooks[0], hooks[1], None) == gedwalk.OK


@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("kw", [dict(precision="fp32"), dict(precision="fp64"), dict(adaptive=True), dict(stochastic=True),
                                dict(lookahead=1, spec_cols=4), dict(L=14)])
def test_charge_covers_what_a_maximisation_allocates(cuda_device, directed, kw):
    from paper_1910_13874_gb300 import gedwalk

    state = {"blocks": {}, "now": 0, "peak": 0}
    counting_allocator(state)
    try:
        G = gedwalk.Graph.from_host(gg.rmat(13, 8, seed=3, directed=directed), directed=directed)
        srv = gedwalk.Server([G], mem_budget=1 << 34)
        state.update(now=0, peak=0)
        srv.poll(srv.submit_maximize(0, 10, **kw))
        charged = srv.stats()["peak_bytes"]
        srv.close()
        G.free()
    finally:
        gedwalk.load().gedwalk_set_allocator(gedwalk._ALLOC_FN(), gedwalk._FREE_FN(), None)
        gedwalk._torch_hooks = None
        gedwalk.use_torch_allocator()
    assert 0 < state["peak"] <= charged


@pytest.mark.parametrize("kind", ["plain", "weighted", "directed"])
@pytest.mark.parametrize("L", [4, 9, 15])
def test_charge_covers_what_a_scoring_allocates(cuda_device, kind, L):
    from paper_1910_13874_gb300 import gedwalk

    state = {"blocks": {}, "now": 0, "peak": 0}
    counting_allocator(state)
    try:
        G = gedwalk.Graph.from_host(gg.rmat(13, 8, seed=3, directed=kind == "directed"), directed=kind == "directed",
                                    weighted=kind == "weighted")
        srv = gedwalk.Server([G], mem_budget=1 << 34)
        state.update(now=0, peak=0)
        srv.poll(srv.submit_score(0, [1, 2, 3, 100], L=L))
        charged = srv.stats()["peak_bytes"]
        srv.close()
        G.free()
    finally:
        gedwalk.load().gedwalk_set_allocator(gedwalk._ALLOC_FN(), gedwalk._FREE_FN(), None)
        gedwalk._torch_hooks = None
        gedwalk.use_torch_allocator()
    assert 0 < state["peak"] <= charged
