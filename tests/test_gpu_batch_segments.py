"""The default complex64 trajectory batch (states in shared memory, matrix
entries cut evenly over the CTAs) against the XOR-ELL schedule of the same
batch, for sizes on both sides of the shared-memory limit and down to one
slab of rows, with trajectories that end early."""

import numpy as np
import pytest

import paper_2606_29692_gb300 as tq
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(4,), (8, 4, 6), (16, 4, 14, 10, 12, 16)])
def test_segments_match_xell(sizes):
    ctx = tq.Context(0)
    hams, pools, ne, mp, th = [], [], [], [], []
    rng = np.random.default_rng(9)
    for i, q in enumerate(sizes):
        ints = synth.integrals(q // 2, 300 + i)
        e = max(2, 2 * (q // 4))
        hams.append(tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, i % 2, tq.TQ_C64))
        pools.append(tq.build_pool(ctx, q // 2, e, i % 2))
        ne.append(e)
        mp.append(i % 2)
        th.append(rng.normal(0, 0.1, size=1 + (5 * i) % 7))
    b = tq.Batch(ctx, hams, pools, ne, mp, th, 1e-9)
    b.run(True)
    got, psi = b.results(), [b.state(t) for t in range(len(sizes))]
    b.run(False)                                             # the same launches outside a graph
    for t in range(len(sizes)):
        assert np.array_equal(b.results()[t]["energy"], got[t]["energy"])
        assert np.array_equal(b.state(t), psi[t])
    b.set_schedule(tq.TQ_SPMV_XELL)
    b.run(True)
    want = b.results()
    # rows of at most 360 float32 products, summed in another order: below
    # 360 eps per unit of sum |H_rc psi_c| (at most 10 Ha here)
    tol = 360 * np.finfo(np.float32).eps * 10
    for t in range(len(sizes)):
        assert got[t]["n_iter"] == want[t]["n_iter"]
        assert np.array_equal(got[t]["selected"], want[t]["selected"])
        assert np.abs(got[t]["energy"] - want[t]["energy"]).max() <= tol
        assert np.abs(got[t]["max_grad"] - want[t]["max_grad"]).max() <= tol
        assert np.linalg.norm(psi[t] - b.state(t)) <= 1e-5
