"""ising_batch_get_spins at the sizes where its path changes and around them, the
smallest instances, and in any order of calls."""

import numpy as np
import pytest

import synth
from test_gpu_map import P  # noqa: F401

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 3, 4, 5, 1023, 1024, 1025, 6143, 16385, 40001, 7]


def test_set_and_get(P):  # noqa: F811
    rng = np.random.default_rng(1)
    gs = [synth.er_graph(n, min(1.0, 6 / max(n - 1, 1)), n, "pm1") for n in SIZES]
    spins = [[rng.choice(np.array([-1, 1], np.int8), n) for _ in range(3)] for n in SIZES]
    with P.ising_batch_create([(g.n, g.src, g.dst, g.w) for g in gs], replicas=3) as b:
        for k in range(len(gs)):
            for r in range(3):
                P.ising_batch_set_spins(b, k, r, spins[k][r])
        for k in list(range(len(gs))) + list(reversed(range(len(gs)))):
            for r in range(3):
                assert np.array_equal(P.ising_batch_get_spins(b, k, r), spins[k][r]), (SIZES[k], r)


def test_a_replayed_anneal_that_timed_out(P):  # noqa: F811
    import torch
    g = synth.er_graph(20011, 8 / 20010, 1, "pm1")
    small = synth.er_graph(300, 8 / 299, 2, "pm1")
    stream = torch.cuda.Stream()
    with P.ising_batch_create([(x.n, x.src, x.dst, x.w) for x in (g, small)], replicas=2, stream=stream) as b:
        P.ising_batch_init_random(b, 1)
        P.ising_batch_debug_fault(b, P.ISING_FAULT_SKIP_ARRIVAL, 20_000_000)  # 20 ms
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            P.ising_batch_anneal(b, p0=0.1, t_total=10, seed=3, stream=stream)
        P.ising_batch_get_spins(b, 1, 0)
        P.ising_batch_get_spins(b, 1, 0)
        with torch.cuda.stream(stream):
            graph.replay()
        with pytest.raises(P.IsingError) as e:
            P.ising_batch_get_spins(b, 1, 0)
        assert e.value.code == P.ISING_ETIMEOUT
