"""The one-launch ansatz sweeps where their shape has more to it than one pair
per thread: several pairs per thread (16 qubits), 1024-thread blocks (18 qubits,
complex64), and state and adjoint vector handed from launch to launch by a
cluster of several blocks (12 qubits, 150 factors).  States against the batched
update, bit for bit; gradients against the launches per factor that sector
spaces and 18-qubit complex128 states take, and against the oracle."""

import numpy as np
import pytest
import torch

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import to_state
from oracle import adapt, vqe

pytestmark = pytest.mark.gpu

EPS = {tq.TQ_C128: np.finfo(np.float64).eps, tq.TQ_C64: np.finfo(np.float32).eps}
DT = {tq.TQ_C128: torch.complex128, tq.TQ_C64: torch.complex64}


def factors(pool, count, seed):
    """Ops with the first and the last of the pool (a single, a double) among them, and angles."""
    rng = np.random.default_rng(seed)
    ops = rng.integers(0, pool.M, size=count)
    ops[0], ops[-1] = 0, pool.M - 1
    return ops, rng.normal(0.0, 0.3, size=count)


def one_by_one(ctx, pool, psi, ops, th, prec):
    d = torch.as_tensor(psi).to(DT[prec]).cuda()[None].contiguous()
    for k, t in zip(ops, th):
        tq.evolve_taylor5_batch(ctx, pool, d, torch.tensor([int(k)], dtype=torch.int32, device="cuda"),
                                torch.tensor([float(t)], dtype=torch.float64, device="cuda"), prec=prec)
    torch.cuda.synchronize()
    return d[0].cpu().numpy()


def bound(count, prec, ham_norm):
    # ten roundings a factor and sweep of an amplitude, root mean square, on
    # a state and an adjoint vector of norms 1 and at most 2 |H|, doubled in
    # 2 Re<chi|U' phi>
    return 2 * 2 * ham_norm * np.sqrt(10.0 * 2 * count) * EPS[prec]


@pytest.mark.parametrize("prec", [tq.TQ_C128, tq.TQ_C64])
@pytest.mark.parametrize("mp", [tq.TQ_JW, tq.TQ_BK])
def test_several_pairs_per_thread(mp, prec):
    n, ne, count = 8, 8, 24
    ctx, ints = tq.Context(0), synth.integrals(n, 77)
    pool = tq.build_pool(ctx, n, ne, mp)
    ham = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, mp, prec)
    ops, th = factors(pool, count, 1)
    full = synth.random_state(2 * n, 6)
    out = tq.State(ctx, 2 * n, prec)
    tq.ansatz_energy_grad(ctx, ham, pool, to_state(ctx, full, 2 * n, prec), ops, th, psi_out=out)
    assert np.array_equal(out.numpy().astype(np.complex128), one_by_one(ctx, pool, full, ops, th, prec).astype(np.complex128))
    # a state of the sector, evaluated in the sector by launches per factor
    na, nb = (ne + 1) // 2, ne // 2
    rows = np.asarray(tq.sector_basis(n, na, nb, mp))
    rng = np.random.default_rng(2)
    part = rng.normal(size=rows.size) + 1j * rng.normal(size=rows.size)
    part /= np.linalg.norm(part)
    psi = np.zeros(1 << (2 * n), complex)
    psi[rows] = part
    E, g = tq.ansatz_energy_grad(ctx, ham, pool, to_state(ctx, psi, 2 * n, prec), ops, th)
    h_s = tq.build_hamiltonian_sector(ctx, ints.h, ints.g, 0.0, mp, tq.TQ_C128, na, nb)
    p_s = tq.build_pool_sector(ctx, n, ne, mp, na, nb)
    E_ref, g_ref = tq.ansatz_energy_grad(ctx, h_s, p_s, to_state(ctx, part, 2 * n, tq.TQ_C128, sector=(na, nb)), ops, th)
    norm = np.abs(np.linalg.eigvalsh(ints.h)).sum() * 4       # a spectral scale of H of these integrals, in Ha
    tol = bound(count, prec, norm)
    assert prec == tq.TQ_C64 or np.abs(g_ref).max() > 1e9 * tol
    assert abs(E - E_ref) <= tol and np.abs(g - g_ref).max() <= tol


def test_wide_blocks():
    n, ne, mp, count = 9, 8, tq.TQ_BK, 20
    ctx, ints = tq.Context(0), synth.integrals(n, 78)
    pool = tq.build_pool(ctx, n, ne, mp)
    ops, th = factors(pool, count, 3)
    psi = synth.random_state(2 * n, 6).astype(np.complex64).astype(complex)
    res = []
    for prec in (tq.TQ_C64, tq.TQ_C128):
        ham = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, mp, prec)
        out = tq.State(ctx, 2 * n, prec)
        ctx.trace(True)
        res.append(tq.ansatz_energy_grad(ctx, ham, pool, to_state(ctx, psi, 2 * n, prec), ops, th, psi_out=out))
        names = set(ctx.trace_report())
        ctx.trace(False)
        # complex128 does not fit one cluster: a launch per factor
        assert ("ansatz_forward" in names) == (prec == tq.TQ_C64) and ("ansatz_dot" in names) == (prec == tq.TQ_C128)
        if prec == tq.TQ_C64:
            assert np.array_equal(out.numpy().astype(np.complex64), one_by_one(ctx, pool, psi, ops, th, prec))
    (E, g), (E_ref, g_ref) = res
    tol = bound(count, tq.TQ_C64, np.abs(np.linalg.eigvalsh(ints.h)).sum() * 4)
    assert abs(E - E_ref) <= tol and np.abs(g - g_ref).max() <= tol


@pytest.mark.parametrize("prec", [tq.TQ_C128, tq.TQ_C64])
def test_launches_of_a_long_ansatz(prec):
    n, ne, mp, count = 6, 4, tq.TQ_BK, 150
    ctx, ints = tq.Context(0), synth.integrals(n, 66)
    s = adapt.build_system(ints, ne, mp)
    ham = tq.build_hamiltonian(ctx, ints.h, ints.g, ints.e_const, mp, prec)
    pool = tq.build_pool(ctx, n, ne, mp)
    ops, th = factors(pool, count, 5)
    th *= 0.3
    psi = synth.random_state(2 * n, 3)
    st, out = to_state(ctx, psi, 2 * n, prec), tq.State(ctx, 2 * n, prec)
    E, g = tq.ansatz_energy_grad(ctx, ham, pool, st, ops, th, psi_out=out)
    assert np.array_equal(out.numpy().astype(np.complex128), one_by_one(ctx, pool, psi, ops, th, prec).astype(np.complex128))
    E_ref, g_ref = vqe.energy_and_gradient(s, list(ops), th, psi)
    tol = bound(count, prec, np.abs(s.ham_pauli.c).sum())
    assert abs(E - E_ref) <= tol and np.abs(g - g_ref).max() <= tol
