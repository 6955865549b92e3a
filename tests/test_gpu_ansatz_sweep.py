"""GPU parity of the one-launch ansatz sweeps where their shape changes: one
thread's worth of pairs (4 qubits), a cluster of several CTAs (12 qubits),
and more factors than one launch takes (8 qubits, 150 factors)."""

import numpy as np
import pytest

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import rel_l2, to_state
from oracle import adapt, vqe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [tq.TQ_C128, tq.TQ_C64])
@pytest.mark.parametrize("n,ne,ops_n,mp", [(2, 2, 3, 0), (4, 4, 150, 1), (6, 4, 9, 0)])
def test_sweeps_match_oracle(n, ne, ops_n, mp, prec):
    ints = synth.integrals(n, 60 + n)
    s = adapt.build_system(ints, ne, mp)
    ctx = tq.Context(0)
    ham = tq.build_hamiltonian(ctx, ints.h, ints.g, ints.e_const, mp, prec)
    pool = tq.build_pool(ctx, n, ne, mp)
    rng = np.random.default_rng(8)
    ops, th = rng.integers(0, len(s.pool), size=ops_n), rng.normal(0, 0.1, size=ops_n)
    psi0 = synth.random_state(2 * n, 3)
    st, out = to_state(ctx, psi0, 2 * n, prec), tq.State(ctx, 2 * n, prec)
    E, g = tq.ansatz_energy_grad(ctx, ham, pool, st, ops, th, psi_out=out)
    E_ref, g_ref = vqe.energy_and_gradient(s, list(ops), th, psi0)
    p_ref = vqe.ansatz_state(s, list(ops), th, psi0)
    # every factor rounds each amplitude a few times: (5 products + 5 sums)
    # eps per factor and sweep, on states of norm 1 and chi of at most
    # 2 sum |H terms|
    eps = np.finfo(np.float64 if prec == tq.TQ_C128 else np.float32).eps
    tol, hmax = 20 * (ops_n + 10) * eps, np.abs(s.ham_pauli.c).sum()
    assert rel_l2(out.numpy(), p_ref) <= tol
    assert abs(E - E_ref) <= tol * hmax
    assert np.abs(g - g_ref).max() <= 2 * tol * hmax
    assert np.array_equal(st.numpy(), psi0.astype(np.complex64 if prec == tq.TQ_C64 else np.complex128))
