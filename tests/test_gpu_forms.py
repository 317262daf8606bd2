"""The kernel forms that ran, in the tests that compare the spin-map engine's and
the clustered batch kernel's spins: a plan that is refused falls back to another
engine with the same spins and the same engine code, so the spins cannot tell."""

import numpy as np
import pytest

import oracle
import test_gpu_batch_map
import test_gpu_map
from test_gpu_map import P  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", sorted(test_gpu_map.GRAPHS))
def test_spin_map_forms(P, name):  # noqa: F811
    g = test_gpu_map.GRAPHS[name]()
    kind = "cluster" if name in ("grid_er", "grid_wide") else name.split("_")[0]  # too sparse for the grid
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        assert P.ising_debug_form(h) == (-1, 0)
        P.ising_init_random(h, 1)
        P.ising_anneal(h, p0=0.2, t_total=2, seed=1)
        form, blocks = P.ising_debug_form(h)
        want = {"block": P.ISING_FORM_MAP_BLOCK_STREAM if "stream" in name else P.ISING_FORM_MAP_BLOCK,
                "cluster": P.ISING_FORM_MAP_CLUSTER, "split": P.ISING_FORM_MAP_CLUSTER, "grid": P.ISING_FORM_MAP_GRID}
        assert form == want[kind]
        assert blocks in {"block": (1,), "cluster": (8, 16), "split": (8, 16), "grid": (152,)}[kind]
        assert (P.ising_engine_used(h) == P.ISING_ENGINE_HUB) == (kind == "split")
        # Algorithm 1 runs in the same form, but not over split rows
        P.ising_anneal(h, kind=P.ISING_SCHED_NFLIP, n0=1, t_total=2, seed=1)
        assert P.ising_debug_form(h) == ((P.ISING_FORM_ENGINE, 0) if kind == "split" else (form, blocks))
        P.ising_anneal(h, p0=0.2, t_total=2, seed=1, mode=P.ISING_MODE_RACY)
        assert P.ising_debug_form(h) == (P.ISING_FORM_ENGINE, 0)
        P.ising_set_engine(h, P.ISING_ENGINE_PERSISTENT_GRID)
        P.ising_anneal(h, p0=0.2, t_total=2, seed=1)
        assert P.ising_debug_form(h) == (P.ISING_FORM_ENGINE, 0)


# dense enough for one block on every SM: each row's share of 110 entries
GRID = {"int8": lambda: test_gpu_map._er(100003, 110), "wide": lambda: test_gpu_map._wide(test_gpu_map._er(100003, 110))}


@pytest.mark.parametrize("weights", sorted(GRID))
def test_grid_form_matches_oracle(P, weights):  # noqa: F811
    g = GRID[weights]()
    s0 = oracle.init_spins(g.n, 5)
    q = np.random.default_rng(2).integers(0, 256, g.n).astype(np.uint8)
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        P.ising_set_spins(h, s0)
        P.ising_anneal(h, p0=0.2, t_total=5, sweeps=2, seed=3)
        P.ising_anneal(h, p0=0.2, t_total=5, t_begin=2, seed=3)
        assert P.ising_debug_form(h) == (P.ISING_FORM_MAP_GRID, 152)
        assert np.array_equal(P.ising_get_spins(h), oracle.anneal(g.n, g.src, g.dst, g.w, s0, seed=3, p0=0.2, T=5))
        P.ising_set_spins(h, s0)
        P.ising_anneal(h, kind=P.ISING_SCHED_NFLIP, n0=300, t_total=3, seed=11)
        assert P.ising_debug_form(h) == (P.ISING_FORM_MAP_GRID, 152)
        assert np.array_equal(P.ising_get_spins(h), oracle.anneal_nflip(g.n, g.src, g.dst, g.w, s0, seed=11, n0=300, T=3))
        P.ising_set_flip_bias(h, q)
        P.ising_set_spins(h, s0)
        P.ising_anneal(h, p0=0.3, t_total=3, seed=4)
        want = oracle.anneal(g.n, g.src, g.dst, g.w, s0, seed=4, p0=0.3, T=3, bias=q)
        assert np.array_equal(P.ising_get_spins(h), want)


def test_grid_form_reports_a_silent_block(P):  # noqa: F811
    g = GRID["int8"]()
    for kw in (dict(p0=0.1), dict(kind=P.ISING_SCHED_NFLIP, n0=20)):
        with P.ising_create(g.n, g.src, g.dst, g.w) as h:
            P.ising_debug_fault(h, P.ISING_FAULT_SKIP_ARRIVAL, 50_000_000)  # 50 ms
            P.ising_init_random(h, 1)
            P.ising_anneal(h, t_total=30, seed=3, **kw)
            assert P.ising_debug_form(h) == (P.ISING_FORM_MAP_GRID, 152)
            with pytest.raises(P.IsingError) as e:
                P.ising_cut(h)
            assert e.value.code == P.ISING_ETIMEOUT


# instances on the one-block kernel, and on 1, 2, 4, 8, 16 blocks
BATCHES = {
    "pm1": [0, 4, 1, 1, 0, 1],
    "int8": [0, 3, 0, 1, 0, 1],
    "mixed": [0, 1, 2, 0, 0, 0],
    "one_replica": [0, 1, 0, 0, 1, 0],
    "degree63": [0, 2, 0, 0, 0, 0],
    "degree64": [2, 0, 0, 0, 0, 0],
}


@pytest.mark.parametrize("name", sorted(BATCHES))
def test_batch_forms(P, name):  # noqa: F811
    make, replicas = test_gpu_batch_map.BATCHES[name]
    gs = make()
    with P.ising_batch_create([(g.n, g.src, g.dst, g.w) for g in gs], replicas=replicas) as b:
        assert P.ising_batch_debug_form(b)[0] == -1
        P.ising_batch_init_random(b, 3)
        P.ising_batch_anneal(b, p0=0.2, t_total=2, seed=1)
        assert P.ising_batch_debug_form(b) == BATCHES[name]
        P.ising_batch_set_tuning(b, 256, 1, 0)
        P.ising_batch_anneal(b, p0=0.2, t_total=2, seed=1)
        assert P.ising_batch_debug_form(b) == [len(gs), 0, 0, 0, 0, 0]
