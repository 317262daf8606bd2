"""The spin-map engine's plan is optional: where the device has room for a graph
but not for the plan beside it, the handle is created without one and anneals
with the engines that need none."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available()
    from paper_1807_10750_gb300 import _build
    _build.build()
    import paper_1807_10750_gb300 as P
    return P


def test_no_room_for_the_plan(P):
    import torch
    g = synth.er_graph(100003, 50 / 100002, 7, "int8")
    s0 = oracle.init_spins(g.n, 5)
    want = oracle.anneal(g.n, g.src, g.dst, g.w, s0, seed=3, p0=0.2, T=3)

    def anneal(h):
        P.ising_set_spins(h, s0)
        P.ising_anneal(h, p0=0.2, t_total=3, seed=3)
        return P.ising_get_spins(h)

    free = torch.cuda.mem_get_info()[0]
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        assert np.array_equal(anneal(h), want)  # also loads the kernels
        used = free - torch.cuda.mem_get_info()[0]
    # 5M entries of four bytes: the plan takes more than 20 MB of it, so that 12 MB
    # less is enough for the graph
    assert used > 40 << 20
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - used + (12 << 20), dtype=torch.uint8, device="cuda")
    try:
        with P.ising_create(g.n, g.src, g.dst, g.w) as h:
            assert np.array_equal(anneal(h), want)
    finally:
        del fill
        torch.cuda.empty_cache()
