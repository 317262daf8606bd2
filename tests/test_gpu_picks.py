"""Algorithm 1 on the spin-map engine: the picks' buffer belongs to the handle
and does not change with a call's flips or sweeps, so a call allocates nothing
and a captured one stays valid; calls that need more picks than it holds run in
several launches, with the same spins."""

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


def _er(n, degree):
    return synth.er_graph(n, min(1.0, degree / (n - 1)), n, "int8")


def _nflip(P, h, n0, T, **kw):
    P.ising_anneal(h, kind=P.ISING_SCHED_NFLIP, n0=n0, t_total=T, seed=11, **kw)


@pytest.mark.parametrize("n,n0,T", [(33, 1, 20000), (700, 700, 500), (2001, 2001, 300), (20011, 20011, 21)])
def test_several_launches(P, n, n0, T):
    g = _er(n, 6)
    s0 = oracle.init_spins(n, 5)
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        P.ising_set_spins(h, s0)
        _nflip(P, h, n0, T)
        assert np.array_equal(P.ising_get_spins(h), oracle.anneal_nflip(g.n, g.src, g.dst, g.w, s0, seed=11, n0=n0, T=T))


def test_calls_allocate_nothing(P):
    import torch
    g = _er(4001, 10)
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        _nflip(P, h, 1, 2)
        P.ising_cut(h)
        free = torch.cuda.mem_get_info()[0]
        _nflip(P, h, 4000, 2000)
        P.ising_cut(h)
        assert torch.cuda.mem_get_info()[0] == free


def test_a_captured_call_outlives_a_larger_one(P):
    import torch
    g = _er(2001, 25)
    s0 = oracle.init_spins(g.n, 5)
    want = oracle.anneal_nflip(g.n, g.src, g.dst, g.w, s0, seed=11, n0=20, T=8)
    stream = torch.cuda.Stream()
    with P.ising_create(g.n, g.src, g.dst, g.w, stream=stream) as h:
        P.ising_set_spins(h, s0)
        _nflip(P, h, 20, 8, stream=stream)
        assert np.array_equal(P.ising_get_spins(h), want)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            _nflip(P, h, 20, 8, stream=stream)
        _nflip(P, h, 2000, 3000, stream=stream)
        P.ising_set_spins(h, s0)
        with torch.cuda.stream(stream):
            graph.replay()
        assert np.array_equal(P.ising_get_spins(h), want)
