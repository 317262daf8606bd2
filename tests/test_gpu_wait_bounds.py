"""A launch whose waits run out ends within a wait's budget, however many sweeps
it had left."""

import time

import pytest

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


@pytest.mark.parametrize("kw", [dict(kind=1, n0=20), dict(kind=1, n0=2001), dict(p0=0.1)], ids=["nflip", "nflip_all", "linear"])
def test_a_silent_block_of_a_cluster(P, kw):
    assert P.ISING_SCHED_NFLIP == 1
    g = synth.er_graph(2001, 25 / 2000, 2001, "int8")
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        P.ising_debug_fault(h, P.ISING_FAULT_SKIP_ARRIVAL, 50_000_000)  # 50 ms
        P.ising_init_random(h, 1)
        start = time.monotonic()
        P.ising_anneal(h, t_total=20000, sweeps=10000, seed=3, **kw)
        with pytest.raises(P.IsingError) as e:
            P.ising_cut(h)
        # a few launches of a 50 ms wait and some milliseconds of draws each
        assert time.monotonic() - start < 5.0
        assert e.value.code == P.ISING_ETIMEOUT
