"""Energies of one tick on the same Hamiltonian: groups do form when requests
wait together, and where the arena has no room left for their interleaved states
they run one by one, with the bits each request has alone."""

import numpy as np
import pytest

import paper_2606_29692_gb300 as tq
import synth

pytestmark = pytest.mark.gpu

Q, NE, SESSIONS = 18, 4, 16        # states of 2 MiB: half of the smallest budget's 64 MiB


def serve(budget, together):
    """Energies of all sessions after one update each; launches of the interleaving kernel."""
    ctx = tq.Context(0)
    srv = tq.Server(ctx, tq.TQ_C64, hbm_budget=budget, max_batch=64)
    ints = synth.integrals(Q // 2, 91)
    hid = srv.add_hamiltonian(tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, tq.TQ_JW, tq.TQ_C64),
                              tq.build_pool(ctx, Q // 2, NE, tq.TQ_JW))
    for _ in range(SESSIONS):
        srv.add_session(hid, NE, tq.TQ_JW)
    rng = np.random.default_rng(1)
    ops, th = rng.integers(0, 20, size=SESSIONS), rng.normal(0, 0.3, size=SESSIONS)
    script = [(tq.TQ_REQ_EVOLVE, s, int(ops[s]), float(th[s])) for s in range(SESSIONS)]
    script += [(tq.TQ_REQ_ENERGY, s, 0, 0.0) for s in range(SESSIONS)]
    got = []
    if together:                       # all wait in the queue when the loop starts
        for tag, r in enumerate(script):
            srv.submit(*r, tag)
    ctx.trace(True)
    srv.start()
    try:
        if not together:
            for tag, r in enumerate(script):
                srv.submit(*r, tag)
                while len(got) <= tag:
                    got += srv.poll(200000)
        while len(got) < len(script):
            got += srv.poll(200000)
    finally:
        srv.stop()
    packs = ctx.trace_report().get("serve_pack", (0, 0.0))[0]
    ctx.trace(False)
    got.sort(key=lambda c: c["tag"])
    assert all(c["status"] == 0 for c in got)
    return [(c["energy"], c["norm2"]) for c in got], packs


def test_groups_form_and_the_fallback_gives_the_same():
    want, packs = serve(1 << 28, False)
    assert packs == 0                                      # one request a tick
    roomy, packs = serve(1 << 28, True)
    assert packs == 1 and roomy == want                    # one tick of energies
    # the arena's 32 MiB go to the energies' own vectors
    tight, packs = serve(64 << 20, True)
    assert packs == 0 and tight == want
