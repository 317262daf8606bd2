"""The spin-map engine against the CPU oracle, bit for bit, at the sizes where
its forms change: one block (entries resident or streamed), a cluster, the
whole grid; narrow and wide weights, units of 1 to 32 lanes a row, partial
units and single-row classes, graphs with hubs, flip bias, both schedules, resumed runs. And its
bounded waits: a block that sends nothing is reported, not waited for."""

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


def _er(n, degree, seed=1, weights="int8"):
    return synth.er_graph(n, min(1.0, degree / max(n - 1, 1)), seed, weights)


def _wide(g):
    rng = np.random.default_rng(g.n)
    g.w = (rng.integers(1, 1001, g.m) * (2 * rng.integers(0, 2, g.m) - 1)).astype(np.int32)
    return g


def _long_rows():
    # 33 rows of 200 entries beside rows of two
    rng = np.random.default_rng(3)
    ring = np.arange(9001, dtype=np.int32)
    src = np.concatenate([ring, np.repeat(np.arange(33, dtype=np.int32), 200)])
    dst = np.concatenate([np.roll(ring, -1), rng.integers(40, 9001, 33 * 200).astype(np.int32)])
    return synth.Graph(9001, src, dst, synth.draw_weights("int8", src.size, rng))


def _hubs(n, hubs, weights="int8"):
    # rows of 400 to n / 2 drawn ends, a third of them the other hubs', on a cycle
    rng = np.random.default_rng(n + hubs)
    ring = np.arange(n, dtype=np.int32)
    src, dst = [ring], [np.roll(ring, -1)]
    for i in range(hubs):
        d = 400 + (n // 2 - 400) * i // hubs
        src.append(np.full(d, i, np.int32))
        dst.append(np.where((np.arange(d) % 3 == 0) & (hubs > 1), rng.integers(0, hubs, d), rng.integers(hubs, n, d)).astype(np.int32))
    src, dst = np.concatenate(src), np.concatenate(dst)
    keep = src != dst
    return synth.Graph(n, src[keep], dst[keep], synth.draw_weights(weights, int(keep.sum()), rng))


def _star(n):
    src = np.zeros(n - 1, np.int32)
    return synth.Graph(n, src, np.arange(1, n, dtype=np.int32), np.where(np.arange(n - 1) % 3 == 0, 5, -4).astype(np.int32))


GRAPHS = {
    "split_star": lambda: _star(4097),
    "split_one_hub": lambda: _hubs(4100, 1),
    "split_hubs": lambda: _hubs(6000, 17),
    "split_wide": lambda: _wide(_hubs(9001, 60)),
    "split_zipf": lambda: synth.zipf_config_graph(20011, 2.1, 4, 3000, 5),
    "split_zipf_large": lambda: synth.zipf_config_graph(110003, 2.1, 4, 10000, 5),
    "block_n31": lambda: _er(31, 6),
    "block_er800": lambda: _er(800, 48, weights="one"),
    "block_wide": lambda: _wide(_er(500, 20)),
    "block_stream_complete": lambda: synth.complete_graph(200, 1, weights="pm1"),
    "block_stream_dense": lambda: _er(700, 110),
    "cluster_er2001": lambda: _er(2001, 25),
    "cluster_sparse": lambda: _er(8000, 3),
    "cluster_torus": lambda: synth.torus_graph(57, 2, "pm1", Ly=113),
    "cluster_wide": lambda: _wide(_er(9001, 31)),
    "cluster_stream": lambda: _wide(_er(12007, 60)),
    "cluster_dense": lambda: _er(3000, 150),
    "cluster_long_rows": _long_rows,
    "grid_er": lambda: _er(60013, 90),
    "grid_wide": lambda: _wide(_er(80011, 60)),
    "grid_large": lambda: _er(195001, 5),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_matches_oracle(P, name):
    g = GRAPHS[name]()
    s0 = oracle.init_spins(g.n, 5)
    T = 9
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        want = oracle.anneal(g.n, g.src, g.dst, g.w, s0, seed=(7 << 33) | 3, p0=0.2, T=T, replica=2)
        P.ising_set_spins(h, s0)
        P.ising_anneal(h, p0=0.2, t_total=T, sweeps=4, seed=(7 << 33) | 3, replica=2)
        P.ising_anneal(h, p0=0.2, t_total=T, t_begin=4, seed=(7 << 33) | 3, replica=2)
        assert np.array_equal(P.ising_get_spins(h), want)
        # Algorithm 1: the first picks, all vertices but a few, and none
        for n0 in (1, min(g.n, 300), 0):
            want = oracle.anneal_nflip(g.n, g.src, g.dst, g.w, s0, seed=11, n0=n0, T=5)
            P.ising_set_spins(h, s0)
            P.ising_anneal(h, kind=P.ISING_SCHED_NFLIP, n0=n0, t_total=5, seed=11)
            assert np.array_equal(P.ising_get_spins(h), want), n0


@pytest.mark.parametrize("name", ["block_er800", "cluster_er2001", "split_hubs", "grid_er"])
def test_flip_bias(P, name):
    g = GRAPHS[name]()
    s0 = oracle.init_spins(g.n, 5)
    q = np.random.default_rng(2).integers(0, 256, g.n).astype(np.uint8)
    want = oracle.anneal(g.n, g.src, g.dst, g.w, s0, seed=4, p0=0.3, T=6, bias=q)
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        P.ising_set_flip_bias(h, q)
        P.ising_set_spins(h, s0)
        P.ising_anneal(h, p0=0.3, t_total=6, seed=4)
        assert np.array_equal(P.ising_get_spins(h), want)


@pytest.mark.parametrize("name,nflip", [("cluster_er2001", False), ("cluster_er2001", True), ("split_hubs", False),
                                        ("grid_er", False), ("grid_er", True)])
def test_a_silent_block_reports_timeout(P, name, nflip):
    g = GRAPHS[name]()
    kw = dict(kind=P.ISING_SCHED_NFLIP, n0=20) if nflip else dict(p0=0.1)
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        P.ising_debug_fault(h, P.ISING_FAULT_SKIP_ARRIVAL, 50_000_000)  # 50 ms
        P.ising_init_random(h, 1)
        P.ising_anneal(h, t_total=30, seed=3, **kw)
        with pytest.raises(P.IsingError) as e:
            P.ising_cut(h)
        assert e.value.code == P.ISING_ETIMEOUT
    g = _er(300, 15)
    s0 = oracle.init_spins(g.n, 5)
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:  # the context still works
        P.ising_set_spins(h, s0)
        P.ising_anneal(h, p0=0.1, t_total=20, seed=2)
        assert np.array_equal(P.ising_get_spins(h), oracle.anneal(g.n, g.src, g.dst, g.w, s0, seed=2, p0=0.1, T=20))
