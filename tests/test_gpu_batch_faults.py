"""A clustered batch anneal whose waits run out (every block of a cluster waits for
bytes that nobody sends) is reported by whichever call synchronises next, the network's
included, and latched in the batch; a train step on such spins leaves the weights."""

import numpy as np
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


GRAPHS = [synth.er_graph(n, 8 / n, n, "pm1") for n in (20011, 3001, 300)]
N = sum(g.n for g in GRAPHS)


def _batch(P):
    return P.ising_batch_create([(g.n, g.src, g.dst, g.w) for g in GRAPHS], replicas=2)


def _params(P):
    return np.random.default_rng(1).uniform(-0.2, 0.2, P.ISING_GNN_NUM_PARAMS).astype(np.float32)


CALLS = {
    "cuts": lambda P, b, net: P.ising_batch_cuts(b),
    "get_spins": lambda P, b, net: P.ising_batch_get_spins(b, 2, 1),
    "set_spins": lambda P, b, net: P.ising_batch_set_spins(b, 2, 1, np.ones(GRAPHS[2].n, np.int8)),
    "autotune": lambda P, b, net: P.ising_batch_autotune(b, 2),
    "forward": lambda P, b, net: P.ising_gnn_batch_forward(net, b),
    "gradients": lambda P, b, net: P.ising_gnn_batch_gradients(net, b, np.ones(N, np.int8)),
    "train_step": lambda P, b, net: P.ising_gnn_batch_train_step(net, b, np.ones(N, np.int8), 0.01, want_loss=True),
}


@pytest.mark.parametrize("call", sorted(CALLS))
def test_reported_and_latched(P, call):
    params = _params(P)
    net = P.ising_gnn_create(params)
    with _batch(P) as b:
        P.ising_batch_debug_fault(b, P.ISING_FAULT_SKIP_ARRIVAL, 20_000_000)  # 20 ms
        P.ising_batch_init_random(b, 1)
        P.ising_batch_anneal(b, p0=0.1, t_total=30, seed=3)
        if call == "train_step":  # steps that do not wait, and one that does
            P.ising_gnn_batch_train_step(net, b, np.ones(N, np.int8), 0.01)
        for _ in range(2):
            with pytest.raises(P.IsingError) as e:
                CALLS[call](P, b, net)
            assert e.value.code == P.ISING_ETIMEOUT
    # the network goes on with its weights
    assert np.array_equal(P.ising_gnn_get_params(net), params)
    with _batch(P) as b:
        P.ising_batch_init_random(b, 1)
        P.ising_batch_anneal(b, p0=0.1, t_total=30, seed=3)
        for other in sorted(CALLS):
            CALLS[other](P, b, net)
    assert not np.array_equal(P.ising_gnn_get_params(net), params)
    P.ising_gnn_destroy(net)


def test_arguments(P):
    with _batch(P) as b:
        for kind, budget in ((P.ISING_FAULT_SHORT_COPY, 0), (7, 0), (P.ISING_FAULT_NONE, 61 * 10 ** 9)):
            with pytest.raises(P.IsingError) as e:
                P.ising_batch_debug_fault(b, kind, budget)
            assert e.value.code == P.ISING_EINVAL
