"""The complex64 energy that reads each coupled pair of rows once in four of
its mask classes, against the CSR pass over all of them, at the sizes where
the build lays its tables out: 16 qubits (the smallest), 18 qubits (runs that
span many rounds), and an encoding carried by a GF(2) map (other
masks in the top index bits)."""

import numpy as np
import pytest

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import to_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mapping", [(8, tq.TQ_JW), (8, tq.TQ_BK), (8, "linear"), (9, tq.TQ_JW), (9, tq.TQ_BK)])
def test_half_pass_matches_csr_pass(n, mapping):
    ints = synth.integrals(n, 70 + n)
    ctx = tq.Context(0)
    if mapping == "linear":
        mapping = tq.mapping_linear(tq.TQ_BK, tq.pool_sector_basis(n, n, tq.TQ_BK))
    x, _, c = tq.pauli_hamiltonian(ints.h, ints.g, 0.25, mapping)
    ham = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.25, mapping, tq.TQ_C64)
    psi = synth.random_state(2 * n, 11)
    basis = np.zeros(1 << (2 * n), complex)
    basis[(1 << n) - 1] = 1.0
    psis = [psi, psi * 3.0, basis]                       # the energy is a quotient: any norm
    got = [tq.energy(ctx, ham, to_state(ctx, p, 2 * n, tq.TQ_C64)) for p in psis]
    ctx.set_spmv_schedule(8)
    want = [tq.energy(ctx, ham, to_state(ctx, p, 2 * n, tq.TQ_C64)) for p in psis]
    # each off-diagonal row sum is float32: a lane adds at most groups / 8
    # entries in either pass, with a few more roundings where runs end and
    # where partial sums meet; |off-diagonal part| is at most the 1-norm of its
    # coefficients
    x = np.asarray(x)
    off = x != 0
    depth = np.unique(x[off]).size * (1 / 8 + 1 / 8) + 16
    bound = depth * np.finfo(np.float32).eps * np.abs(np.asarray(c))[off].sum()
    assert np.all(np.abs(np.asarray(got) - want) <= bound)
    assert abs(got[2] - want[2]) <= 1e-12 * abs(want[2])     # one determinant: the diagonal alone, float64

