"""Requests of one tick on the same Hamiltonian are evaluated together (one
to four states per pass): each result has the bits it has alone, for every
group size, with two sizes of Hamiltonian in the mix, and with an arena too
small to interleave states."""

import numpy as np
import pytest

import paper_2606_29692_gb300 as tq
import synth

pytestmark = pytest.mark.gpu

SIZES = ((10, 4), (4, 2))


def serve(sessions, script, budget, alone):
    ctx = tq.Context(0)
    srv = tq.Server(ctx, tq.TQ_C64, hbm_budget=budget, max_batch=64)
    ids = []
    for i, (q, ne) in enumerate(SIZES):
        ints = synth.integrals(q // 2, 80 + i)
        ids.append(srv.add_hamiltonian(tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, i, tq.TQ_C64),
                                       tq.build_pool(ctx, q // 2, ne, i)))
    for h in sessions:
        srv.add_session(ids[h], SIZES[h][1], h)
    srv.start()
    got = []
    try:
        for tag, (kind, sess, op, th) in enumerate(script):
            srv.submit(kind, sess, op, th, tag)
            if alone:
                while len(got) <= tag:
                    got += srv.poll(200000)
        while len(got) < len(script):
            got += srv.poll(200000)
    finally:
        srv.stop()
    got.sort(key=lambda c: c["tag"])
    return [{k: c[k] for k in ("status", "energy", "max_grad", "argmax", "norm2")} for c in got]


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8])
def test_groups_give_single_results(n):
    rng = np.random.default_rng(n)
    sessions = [0] * n + [1] * 2
    script = []
    for r in range(3):
        for s in range(len(sessions)):
            script.append((tq.TQ_REQ_EVOLVE, s, int(rng.integers(0, 2)), float(rng.normal(0, 0.3))))
        for s in range(len(sessions)):
            script.append((int(rng.choice([tq.TQ_REQ_ENERGY, tq.TQ_REQ_GRADIENTS])), s, 0, 0.0))
    want = serve(sessions, script, 1 << 28, True)
    assert all(c["status"] == 0 for c in want)
    assert serve(sessions, script, 1 << 28, False) == want
