"""The form a graph gets, where the choice matters: graphs that the spin-map
engine's forms were slower on than the engines that need no map keep those. Spins
do not depend on it."""

import numpy as np
import pytest

import oracle
import synth
from test_gpu_map import P  # noqa: F401

pytestmark = pytest.mark.gpu


def _er(n, degree):
    return synth.er_graph(n, degree / (n - 1), 3, "pm1")


# graph, form of a call of several sweeps (of item dataflow for the lattices), of
# one sweep, and of several with Algorithm 1's flips
GRAPHS = {
    "near_clique": (lambda: synth.complete_graph(800, 1, weights="pm1"), "ENGINE", "ENGINE", "ENGINE"),
    "two_class_lattice_small": (lambda: synth.torus_graph(140, 2, "pm1"), "MAP_CLUSTER", "MAP_CLUSTER", "MAP_CLUSTER"),
    "two_class_lattice": (lambda: synth.torus_graph(270, 2, "pm1", Ly=260), "MAP_CLUSTER", "ENGINE", "MAP_CLUSTER"),
    "two_class_lattice_large": (lambda: synth.torus_graph(300, 2, "pm1"), "ENGINE", "ENGINE", "MAP_CLUSTER"),
    "odd_lattice": (lambda: synth.torus_graph(301, 2, "pm1"), "MAP_CLUSTER", "ENGINE", "MAP_CLUSTER"),
    "sparse": (lambda: _er(150011, 4), "MAP_CLUSTER", "ENGINE", "MAP_CLUSTER"),
    "sparse_small": (lambda: _er(50021, 6), "MAP_CLUSTER", "MAP_CLUSTER", "MAP_CLUSTER"),
    "denser": (lambda: _er(130003, 20), "MAP_CLUSTER", "MAP_CLUSTER", "MAP_CLUSTER"),
    "sparse_large": (lambda: _er(200003, 4), "ENGINE", "ENGINE", "ENGINE"),
    "six_large": (lambda: _er(200003, 6), "MAP_GRID", "ENGINE", "MAP_GRID"),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_forms_and_spins(P, name):  # noqa: F811
    make, several, one, nflip = GRAPHS[name]
    g = make()
    s0 = oracle.init_spins(g.n, 5)
    with P.ising_create(g.n, g.src, g.dst, g.w) as h:
        P.ising_set_spins(h, s0)
        if "lattice" in name:
            P.ising_set_engine(h, P.ISING_ENGINE_ITEMFLOW)
        for t, sweeps, form in ((0, 3, several), (3, 1, one), (4, 2, several)):
            P.ising_anneal(h, p0=0.2, t_total=6, t_begin=t, sweeps=sweeps, seed=3)
            assert P.ising_debug_form(h)[0] == getattr(P, "ISING_FORM_" + form), (t, sweeps)
        assert np.array_equal(P.ising_get_spins(h), oracle.anneal(g.n, g.src, g.dst, g.w, s0, seed=3, p0=0.2, T=6))
        P.ising_set_engine(h, P.ISING_ENGINE_AUTO)
        P.ising_set_spins(h, s0)
        for t, sweeps, form in ((0, 2, nflip), (2, 1, one), (3, 2, nflip)):
            P.ising_anneal(h, kind=P.ISING_SCHED_NFLIP, n0=200, t_total=5, t_begin=t, sweeps=sweeps, seed=11)
            assert P.ising_debug_form(h)[0] == getattr(P, "ISING_FORM_" + form), (t, sweeps)
        assert np.array_equal(P.ising_get_spins(h), oracle.anneal_nflip(g.n, g.src, g.dst, g.w, s0, seed=11, n0=200, T=5))
