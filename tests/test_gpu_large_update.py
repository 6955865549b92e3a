"""The two-launch update of a state beyond one thread-block cluster (18
qubits: the smallest such size for either precision is 17), against the
batched full-state update of the same state and a float64 normalisation;
and inside an ADAPT step."""

import numpy as np
import pytest
import torch

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import rel_l2, to_state

pytestmark = pytest.mark.gpu

Q, NE = 18, 4


@pytest.fixture(scope="module")
def setup():
    ctx = tq.Context(0)
    return ctx, tq.build_pool(ctx, Q // 2, NE, tq.TQ_BK), 1.7 * synth.random_state(Q, 12)


def batched(ctx, pool, psi, k, th, prec):
    d = torch.as_tensor(psi).to(torch.complex64 if prec == tq.TQ_C64 else torch.complex128).cuda()[None].contiguous()
    tq.evolve_taylor5_batch(ctx, pool, d, torch.tensor([k], dtype=torch.int32, device="cuda"),
                            torch.tensor([th], dtype=torch.float64, device="cuda"), prec=prec)
    torch.cuda.synchronize()
    return d[0].cpu().numpy().astype(np.complex128)


@pytest.mark.parametrize("prec", [tq.TQ_C128, tq.TQ_C64])
@pytest.mark.parametrize("pick,th", [(0, 0.4), (0.5, -0.07), (1, 1.3)])
def test_update_and_norm(setup, pick, th, prec):
    ctx, pool, psi = setup
    k = int(pick * (pool.M - 1))
    ref = batched(ctx, pool, psi, k, th, prec)
    eps = np.finfo(np.float64 if prec == tq.TQ_C128 else np.float32).eps
    for renorm in (False, True):
        st = to_state(ctx, psi, Q, prec)
        tq.evolve_taylor5(ctx, pool, k, th, st, renormalize=renorm)
        want = ref / np.linalg.norm(ref) if renorm else ref
        # same products; the rescale rounds each amplitude once more, and the
        # float32 sums of 16 squares average over 2^18 amplitudes
        assert rel_l2(st.numpy(), want) <= 4 * eps


def test_adapt_step(setup):
    ctx, pool, psi = setup
    ints = synth.integrals(Q // 2, 5)
    ham = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, tq.TQ_BK, tq.TQ_C64)
    st = to_state(ctx, psi / np.linalg.norm(psi), Q, tq.TQ_C64)
    before = st.numpy()
    r = tq.adapt_step(ctx, ham, pool, st, 1e-9, 0.3)
    ref = batched(ctx, pool, before, r["selected"], 0.3, tq.TQ_C64)
    assert rel_l2(st.numpy(), ref / np.linalg.norm(ref)) <= 4 * np.finfo(np.float32).eps
