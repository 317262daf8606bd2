"""The clustered batch kernel against the CPU oracle, every instance and
replica: one launch per cluster size (a 20,011-vertex instance on 16 blocks
beside single vertices), partial units and empty classes of a block, one to
eight replicas, +-1 and wider weights (also mixed in one batch), the largest
degree it takes and the first that it leaves to the one-block kernel."""

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


def _er(n, degree, seed, weights):
    return synth.er_graph(n, min(1.0, degree / max(n - 1, 1)), seed, weights)


def _star(leaves, extra):
    # one row of `leaves` entries, and a path
    n = leaves + extra
    src = np.concatenate([np.zeros(leaves, np.int32), np.arange(1, n - 1, dtype=np.int32)])
    dst = np.concatenate([np.arange(1, leaves + 1, dtype=np.int32), np.arange(2, n, dtype=np.int32)])
    return synth.Graph(n, src, dst, synth.draw_weights("pm1", src.size, np.random.default_rng(n)))


EDGELESS = synth.Graph(7, np.zeros(0, np.int32), np.zeros(0, np.int32), np.zeros(0, np.int32))


BATCHES = {
    "pm1": (lambda: [_er(n, 10, n, "pm1") for n in (20011, 4001, 1537, 640, 33, 2)] + [EDGELESS], 8),
    "int8": (lambda: [_er(n, 9, n, "int8") for n in (20011, 3001, 129, 32, 31)], 5),
    "mixed": (lambda: [_er(2500, 12, 1, "one"), _er(2600, 30, 2, "int8"), _er(300, 6, 3, "pm1")], 3),
    "one_replica": (lambda: [_er(6001, 6, 1, "one"), _er(500, 40, 2, "one")], 1),
    "many_small": (lambda: [_er(17 + 3 * k, 5, k, "pm1") for k in range(400)], 2),
    "degree63": (lambda: [_star(63, 70), _er(1000, 8, 1, "pm1")], 8),
    "degree64": (lambda: [_star(64, 70), _er(1000, 8, 1, "pm1")], 8),
}


@pytest.mark.parametrize("name", sorted(BATCHES))
def test_matches_oracle(P, name):
    make, replicas = BATCHES[name]
    gs = make()
    T, seed = 7, (5 << 32) | 9
    with P.ising_batch_create([(g.n, g.src, g.dst, g.w) for g in gs], replicas=replicas) as b:
        P.ising_batch_init_random(b, 3)
        P.ising_batch_anneal(b, p0=0.2, t_total=T, sweeps=3, seed=seed)
        P.ising_batch_anneal(b, p0=0.2, t_total=T, t_begin=3, seed=seed)
        cuts = P.ising_batch_cuts(b)
        for k, g in enumerate(gs):
            if len(gs) > 20 and k % 37:
                continue
            for r in range(replicas):
                s0 = oracle.init_spins(g.n, 3, instance=k, replica=r)
                want = oracle.anneal(g.n, g.src, g.dst, g.w, s0, seed=seed, p0=0.2, T=T, instance=k, replica=r)
                assert np.array_equal(P.ising_batch_get_spins(b, k, r), want), (k, r)
                assert cuts[k, r] == oracle.energy_cut(g.n, g.src, g.dst, g.w, want)[2]
        P.ising_batch_autotune(b, 3)  # goes on from the same spins, whichever form it keeps
        assert np.array_equal(P.ising_batch_cuts(b), cuts)
