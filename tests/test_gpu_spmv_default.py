"""The H pass's schedule: kept per precision, back to the default, and a tuned
context no slower than an untuned one (every default is one of the schedules
that the tuner times, and the energy alone stays on its own pass)."""

import pytest

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import to_state

pytestmark = pytest.mark.gpu


def problem(ctx, n, prec, ne=4):
    ints = synth.integrals(n, 30 + n)
    return (tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, tq.TQ_BK, prec), tq.build_pool(ctx, n, ne, tq.TQ_BK),
            to_state(ctx, synth.random_state(2 * n, 2), 2 * n, prec))


def passes(ctx, ham, pool, st):
    """Launch names of the H pass of the gradients, and the gradients."""
    ctx.trace(True)
    g = tq.pool_gradients(ctx, ham, pool, st)
    names = set(ctx.trace_report())
    ctx.trace(False)
    return names & {"energy_csr", "energy_xell"}, g.tolist()


def test_tuning_one_precision_leaves_the_other():
    ctx = tq.Context(0)
    small, large = problem(ctx, 6, tq.TQ_C128), problem(ctx, 6, tq.TQ_C64)
    want = passes(ctx, *large)
    assert want[0] == {"energy_xell"}
    tq.autotune_spmv(ctx, small[0], small[2])
    assert passes(ctx, *large) == want


@pytest.mark.parametrize("n,lanes", [(6, 16), (7, 8), (8, 4)])
def test_default_of_complex128_is_among_the_schedules(n, lanes):
    ctx = tq.Context(0)
    p = problem(ctx, n, tq.TQ_C128)
    want = passes(ctx, *p)
    ctx.set_spmv_schedule(lanes)
    assert passes(ctx, *p) == want


@pytest.mark.parametrize("prec", [tq.TQ_C128, tq.TQ_C64])
def test_back_to_the_default(prec):
    ctx = tq.Context(0)
    p = problem(ctx, 7, prec)
    want = passes(ctx, *p), tq.energy(ctx, p[0], p[2])
    ctx.set_spmv_schedule(32 if prec == tq.TQ_C64 else tq.TQ_SPMV_XELL)
    assert passes(ctx, *p)[0] != want[0][0]
    ctx.set_spmv_schedule(tq.TQ_SPMV_AUTO)
    assert (passes(ctx, *p), tq.energy(ctx, p[0], p[2])) == want
    for bad in (-2, 1, 5, 64):
        with pytest.raises(tq.TQError):
            ctx.set_spmv_schedule(bad)


def test_energy_alone_after_tuning():
    ctx = tq.Context(0)
    ham, _, st = problem(ctx, 8, tq.TQ_C64)
    want = tq.energy(ctx, ham, st)
    tq.autotune_spmv(ctx, ham, st)
    assert tq.energy(ctx, ham, st) == want
    ctx.set_spmv_schedule(8)                    # asked for: the CSR
    assert tq.energy(ctx, ham, st) != want
