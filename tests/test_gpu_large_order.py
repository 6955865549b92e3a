"""Updates of a state beyond one thread-block cluster in a row, where each
launch overlaps the one before: unsynchronised calls against synchronised
ones, and graph-replayed ADAPT runs (line search, norm, update, record in a
chain) against single steps, also past convergence, bit for bit."""

import numpy as np
import pytest
import torch

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import to_state

pytestmark = pytest.mark.gpu

Q, NE, N = 18, 4, 6


@pytest.fixture(scope="module")
def setup():
    ctx = tq.Context(0)
    return ctx, tq.build_pool(ctx, Q // 2, NE, tq.TQ_BK)


@pytest.mark.parametrize("prec", [tq.TQ_C128, tq.TQ_C64])
@pytest.mark.parametrize("renorm", [True, False])
def test_unsynchronised_updates(setup, prec, renorm):
    ctx, pool = setup
    rng = np.random.default_rng(3)
    ops, th = rng.integers(0, pool.M, size=24), rng.normal(0.0, 0.4, size=24)
    psi = 0.7 * synth.random_state(Q, 5)
    out = []
    for sync in (True, False):
        st = to_state(ctx, psi, Q, prec)
        torch.cuda.synchronize()
        for k, t in zip(ops, th):
            tq.evolve_taylor5(ctx, pool, int(k), float(t), st, renormalize=renorm)
            if sync:
                torch.cuda.synchronize()
        out.append(st.numpy())
    assert np.array_equal(*out)


@pytest.mark.parametrize("prec", [tq.TQ_C128, tq.TQ_C64])
@pytest.mark.parametrize("given", [False, True])
def test_run_equals_steps(setup, prec, given):
    ctx, pool = setup
    ints = synth.integrals(Q // 2, 5)
    ham = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, tq.TQ_BK, prec)
    thetas = np.random.default_rng(5).normal(0.0, 0.1, size=N) if given else None
    a = tq.State(ctx, Q, prec)
    tq.state_set_hf(a, NE, tq.TQ_BK)
    ref, states = [], [a.numpy()]
    for i in range(N):
        ref.append(tq.adapt_step(ctx, ham, pool, a, 1e-9, float(thetas[i]) if given else float("nan")))
        states.append(a.numpy())
    # to the end, and with a bound that the smallest gradient meets first
    grads = [r["max_grad"] for r in ref]
    j = int(np.argmin(grads))
    assert j > 0 or given                      # the line search converges part of the way
    for eps, last in ((1e-9, N), (np.nextafter(grads[j], np.inf), j)):
        b = tq.State(ctx, Q, prec)
        tq.state_set_hf(b, NE, tq.TQ_BK)
        got, done = tq.adapt_run(ctx, ham, pool, b, eps, N, thetas)
        assert done == min(last + 1, N)
        assert got[:last] == ref[:last]
        assert np.array_equal(b.numpy(), states[last])
        for g in got[last:]:
            assert g["converged"] and (g["energy"], g["max_grad"]) == (ref[last]["energy"], ref[last]["max_grad"])
