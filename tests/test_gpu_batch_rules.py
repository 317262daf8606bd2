"""Which instances of a batch run in the clustered form and which on the one-block
kernel, and that both side by side give the oracle's spins."""

import numpy as np
import pytest

import oracle
import synth
from test_gpu_map import P  # noqa: F401

pytestmark = pytest.mark.gpu


def _er(n, degree, seed, weights="pm1"):
    return synth.er_graph(n, min(1.0, degree / (n - 1)), seed, weights)


def _small(count, n=60):
    base = [_er(n + k, 8, k) for k in range(20)]
    return [base[k % 20] for k in range(count)]


# instances on the one-block kernel, and in the clustered form on 1, 2, 4, 8, 16 blocks
BATCHES = {
    "two_an_sm": (lambda: _small(300), 8, [0, 300, 0, 0, 0, 0]),
    "many_small": (lambda: _small(400), 8, [400, 0, 0, 0, 0, 0]),
    "many_beside_large": (lambda: [_er(20011, 8, 1)] + _small(400) + [_er(2500, 8, 2)], 3, [400, 0, 1, 0, 0, 1]),
    "few_beside_large": (lambda: [_er(20011, 8, 1)] + _small(200), 8, [0, 200, 0, 0, 0, 1]),
    "many_of_1000": (lambda: [_er(1000, 8, k % 4) for k in range(400)], 8, [0, 400, 0, 0, 0, 0]),
    "many_of_1000_one_replica": (lambda: [_er(1000, 8, k % 4) for k in range(400)], 1, [400, 0, 0, 0, 0, 0]),
    "cliques": (lambda: [synth.complete_graph(60, 1, weights="pm1")] * 300, 2, [300, 0, 0, 0, 0, 0]),
    "small_cliques": (lambda: [synth.complete_graph(20, 1, weights="pm1")] * 300, 2, [0, 300, 0, 0, 0, 0]),
}


@pytest.mark.parametrize("name", sorted(BATCHES))
def test_forms_and_spins(P, name):  # noqa: F811
    make, replicas, forms = BATCHES[name]
    gs = make()
    T, seed = 6, (5 << 32) | 9
    with P.ising_batch_create([(g.n, g.src, g.dst, g.w) for g in gs], replicas=replicas) as b:
        P.ising_batch_init_random(b, 3)
        P.ising_batch_anneal(b, p0=0.2, t_total=T, sweeps=2, seed=seed)
        P.ising_batch_anneal(b, p0=0.2, t_total=T, t_begin=2, seed=seed)
        assert P.ising_batch_debug_form(b) == forms
        cuts = P.ising_batch_cuts(b)
        for k, g in enumerate(gs):
            if k % 29 and g.n < 2000:
                continue
            for r in range(0, replicas, 2):
                s0 = oracle.init_spins(g.n, 3, instance=k, replica=r)
                want = oracle.anneal(g.n, g.src, g.dst, g.w, s0, seed=seed, p0=0.2, T=T, instance=k, replica=r)
                assert np.array_equal(P.ising_batch_get_spins(b, k, r), want), (k, r)
                assert cuts[k, r] == oracle.energy_cut(g.n, g.src, g.dst, g.w, want)[2]
        # another form goes on from the same spins
        P.ising_batch_anneal(b, p0=0.2, t_total=T, seed=7)
        want = P.ising_batch_cuts(b)
        P.ising_batch_init_random(b, 3)
        P.ising_batch_set_tuning(b, 128, 1, 32)
        for t, sweeps, s in ((0, T, seed), (0, T, 7)):
            P.ising_batch_anneal(b, p0=0.2, t_total=T, t_begin=t, sweeps=sweeps, seed=s)
        assert P.ising_batch_debug_form(b) == [len(gs), 0, 0, 0, 0, 0]
        assert np.array_equal(P.ising_batch_cuts(b), want)
