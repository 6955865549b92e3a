"""Calls of different sizes on two threads at once, each with its own context:
what a launch may use of shared memory is a property of the kernel, which both
share."""

import threading

import numpy as np
import pytest

import paper_2606_29692_gb300 as tq
import synth

pytestmark = pytest.mark.gpu


def build(n):
    ctx, ints = tq.Context(0), synth.integrals(n, 50 + n)
    return lambda: tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, tq.TQ_JW, tq.TQ_C128).nnz


def ansatz(n):
    ctx, ints, ne = tq.Context(0), synth.integrals(n, 50 + n), 2
    ham = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, tq.TQ_JW, tq.TQ_C128)
    pool, st = tq.build_pool(ctx, n, ne, tq.TQ_JW), tq.State(ctx, 2 * n, tq.TQ_C128)
    tq.state_set_hf(st, ne, tq.TQ_JW)
    ops, th = np.arange(3) % pool.M, np.full(3, 0.1)
    return lambda: tq.ansatz_energy_grad(ctx, ham, pool, st, ops, th)[0]


@pytest.mark.parametrize("make,reps", [(build, 400), (ansatz, 2000)])
def test_sizes_side_by_side(make, reps):
    calls = [make(2), make(7)]
    want = [c() for c in calls]
    bad, done = [], threading.Event()

    def small():
        try:
            while not done.is_set():
                if calls[0]() != want[0]:
                    bad.append("small: another result")
        except tq.TQError as e:
            bad.append(f"small: {e}")

    t = threading.Thread(target=small)
    t.start()
    try:
        for _ in range(reps):
            assert calls[1]() == want[1]
    finally:
        done.set()
        t.join()
    assert not bad, bad[:3]
