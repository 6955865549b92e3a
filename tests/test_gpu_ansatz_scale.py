"""Energy and gradient of an ansatz do not depend on the norm of the state it
starts from: scaled by a power of two that leaves every amplitude well inside
float32's range, each bit stays.  (Products of two amplitudes leave that range;
they are float64, or taken of a scaled adjoint vector.)"""

import numpy as np
import pytest

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import to_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [tq.TQ_C128, tq.TQ_C64])
@pytest.mark.parametrize("n,ops_n", [(4, 6), (6, 140)])
def test_power_of_two_scaling(n, ops_n, prec):
    ctx, ints, ne = tq.Context(0), synth.integrals(n, 60 + n), 4
    ham = tq.build_hamiltonian(ctx, ints.h, ints.g, ints.e_const, tq.TQ_BK, prec)
    pool = tq.build_pool(ctx, n, ne, tq.TQ_BK)
    rng = np.random.default_rng(1)
    ops, th = rng.integers(0, pool.M, size=ops_n), rng.normal(0, 0.1, size=ops_n)
    psi = synth.random_state(2 * n, 3)
    psi = psi.astype(np.complex64).astype(complex)
    want = tq.ansatz_energy_grad(ctx, ham, pool, to_state(ctx, psi, 2 * n, prec), ops, th)
    assert np.abs(want[1]).max() > 1e-3
    for k in (-70, -40, 40, 60):
        E, g = tq.ansatz_energy_grad(ctx, ham, pool, to_state(ctx, psi * 2.0 ** k, 2 * n, prec), ops, th)
        assert E == want[0] and np.array_equal(g, want[1]), k
