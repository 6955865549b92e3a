"""GPU parity of the table-driven full-space Hamiltonian build at the sizes
where its blocks, segments and table kinds change: 4 qubits (two row blocks,
no wide group), 6 and 10 qubits (one and two table runs per wide group), and
an encoding carried by a GF(2) map (other ranks in the low index bits)."""

import numpy as np
import pytest

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import ham_csr_numpy, oracle_split
from oracle import pauli

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [tq.TQ_C128, tq.TQ_C64])
@pytest.mark.parametrize("n", [2, 3, 5])
@pytest.mark.parametrize("mapped", [False, True])
def test_build_matches_oracle(n, mapped, prec):
    ints = synth.integrals(n, 40 + n)
    ctx = tq.Context(0)
    ps = pauli.qubit_hamiltonian(ints.h, ints.g, 0.25, tq.TQ_BK)
    H = pauli.pauli_to_csr(ps)
    mapping = tq.TQ_BK
    if mapped:
        rows = tq.pool_sector_basis(n, 2, tq.TQ_BK)
        mapping = tq.mapping_linear(tq.TQ_BK, rows)
        old = np.argsort(tq.linear_index(rows))       # base index of each new index
        H = H[old][:, old]
    ham = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.25, mapping, prec)
    rowptr, col, val, diag = ham_csr_numpy(ham)
    orp, ocol, oval, odiag = oracle_split(H)
    assert np.array_equal(rowptr, orp) and np.array_equal(col, ocol)
    # a value is a sum of at most 2 n + 6 terms of at most maxc each: rounding
    # of either side stays below (2 n + 6)^2 eps maxc, in float32 one more
    # rounding of the value itself
    maxc = np.abs(ps.c).max()
    bound = (2 * n + 6) ** 2 * np.finfo(np.float64).eps * maxc
    if prec == tq.TQ_C64:
        bound = bound + np.finfo(np.float32).eps * np.abs(oval)
    assert np.all(np.abs(val.astype(np.float64) - oval) <= bound)
    assert np.abs(diag - odiag).max() <= ps.c.size * np.finfo(np.float64).eps * np.abs(ps.c).sum()
