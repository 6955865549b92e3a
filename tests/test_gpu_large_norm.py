"""How far from 1 a renormalised complex64 state beyond one thread-block
cluster ends up.  The norm is that of the updated amplitudes as rounded and the
factor is applied with more digits than float32, so only zero-mean roundings
remain: at most 24 in a thread's plain sum of 16 squares, and one per
amplitude in the rescale."""

import numpy as np
import pytest

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import to_state

pytestmark = pytest.mark.gpu

Q = 18


@pytest.mark.parametrize("scale,pick,th", [(1.7, 0.0, 0.4), (0.9, 0.5, -0.07), (3.1, 1.0, 1.3), (0.6, 0.3, -0.9),
                                           (1.3, 0.8, 0.02), (2.3, 0.6, 0.6)])
def test_norm_after_rescale(scale, pick, th):
    ctx = tq.Context(0)
    pool = tq.build_pool(ctx, Q // 2, 4, tq.TQ_JW)
    st = to_state(ctx, scale * synth.random_state(Q, 21), Q, tq.TQ_C64)
    tq.evolve_taylor5(ctx, pool, int(pick * (pool.M - 1)), th, st, renormalize=True)
    got = st.numpy()
    norm = np.sqrt(np.sum(got.real.astype(np.longdouble) ** 2 + got.imag.astype(np.longdouble) ** 2))
    # a rounding has relative size 2^-24 / sqrt(3) (root mean square), threads
    # of 8 amplitudes are independent, |psi_i|^2 of a random state spreads like
    # its mean; the norm takes half the error of its square; six deviations
    D, u = 1 << Q, 2.0 ** -24
    sums = 0.5 * np.sqrt(24 / 3) / np.sqrt(D / 8)
    rescale = np.sqrt(2 / 3 / D)
    assert abs(norm - 1) <= 6 * u * (sums + rescale)


def test_norm_below_the_range():
    """Squares below float32's range: the factor is infinite, as it is for the batched update's norm."""
    ctx = tq.Context(0)
    pool = tq.build_pool(ctx, Q // 2, 4, tq.TQ_JW)
    psi = np.zeros(1 << Q, complex)
    psi[5], psi[9] = 1e-30, -1e-30j
    st = to_state(ctx, psi, Q, tq.TQ_C64)
    tq.evolve_taylor5(ctx, pool, 0, 0.0, st, renormalize=True)
    got = st.numpy()
    assert got[5].real == np.inf and got[9].imag == -np.inf
    assert np.all(np.isnan(got[[5, 9]].view(float)[[1, 2]])) and np.all(np.isnan(got[10:20]))
