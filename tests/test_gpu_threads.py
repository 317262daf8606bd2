"""Handles of different sizes in threads of their own: kernels that several
handles share take launches of every size at any time, so no handle's calls fail
or change another's spins."""

import threading

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


def _er(n, degree, weights="one"):
    return synth.er_graph(n, min(1.0, degree / (n - 1)), n, weights)


def _in_threads(jobs):
    errors = []

    def run(job):
        try:
            job()
        except BaseException as e:  # noqa: BLE001 -- reported below
            errors.append(e)

    threads = [threading.Thread(target=run, args=(job,)) for job in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


def test_graphs_of_different_sizes(P):
    import torch

    def job(n, calls):
        g = _er(n, 48)
        want = oracle.anneal(g.n, g.src, g.dst, g.w, oracle.init_spins(g.n, 5), seed=3, p0=0.2, T=calls)
        stream = torch.cuda.Stream()
        for _ in range(3):  # creating a handle looks at its kernel's limits too
            with P.ising_create(g.n, g.src, g.dst, g.w, stream=stream) as h:
                P.ising_init_random(h, 5)
                for t in range(calls):
                    P.ising_anneal(h, p0=0.2, t_total=calls, t_begin=t, sweeps=1, seed=3, stream=stream)
                assert np.array_equal(P.ising_get_spins(h), want), n

    _in_threads([lambda n=n: job(n, 700) for n in (800, 300, 650, 450)])


def test_batches_of_different_sizes(P):
    import torch

    def job(n, calls):
        gs = [_er(n, 4, "pm1"), _er(n // 2, 4, "pm1")]
        want = oracle.anneal(gs[0].n, gs[0].src, gs[0].dst, gs[0].w,
                             oracle.init_spins(gs[0].n, 5, instance=0, replica=1), seed=3, p0=0.2, T=calls, instance=0,
                             replica=1)
        stream = torch.cuda.Stream()
        with P.ising_batch_create([(g.n, g.src, g.dst, g.w) for g in gs], replicas=2, stream=stream) as b:
            P.ising_batch_init_random(b, 5)
            for t in range(calls):
                P.ising_batch_anneal(b, p0=0.2, t_total=calls, t_begin=t, sweeps=1, seed=3, stream=stream)
            assert np.array_equal(P.ising_batch_get_spins(b, 0, 1), want), n
            for t in range(3000):
                P.ising_batch_anneal(b, p0=0.2, t_total=1, seed=t, stream=stream)
            P.ising_batch_cuts(b)

    _in_threads([lambda n=n: job(n, 200) for n in (120000, 60000, 90000, 70000)])
