"""The complex64 energy that reads four of its mask classes from one side
only, where an entry left out, or counted once instead of twice, shows: pairs
of determinants coupled through one mask of every class against float64; and
its rounding on correlated states against that of the pass over all entries."""

import numpy as np
import pytest
import torch

import paper_2606_29692_gb300 as tq
import synth
from gpu_util import to_state

pytestmark = pytest.mark.gpu


def value_at(x, z, c, mask, cols):
    """H[col ^ mask][col] of sum_t c_t X^x Z^z."""
    t = x == mask
    return (1 - 2 * (np.bitwise_count(cols[:, None] & z[t]).astype(int) & 1)) @ c[t]


@pytest.mark.parametrize("n,mapping", [(8, tq.TQ_JW), (8, tq.TQ_BK), (8, "linear"), (9, tq.TQ_JW), (9, tq.TQ_BK)])
def test_every_class_counts(n, mapping):
    ints = synth.integrals(n, 70 + n)
    ctx = tq.Context(0)
    if mapping == "linear":
        mapping = tq.mapping_linear(tq.TQ_BK, tq.pool_sector_basis(n, n, tq.TQ_BK))
    x, z, c = (np.asarray(v) for v in tq.pauli_hamiltonian(ints.h, ints.g, 0.25, mapping))
    x, z = x.astype(np.int64), z.astype(np.int64)
    h64 = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.25, mapping, tq.TQ_C64)
    h128 = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.25, mapping, tq.TQ_C128)
    rng = np.random.default_rng(n)
    masks = np.unique(x[x != 0])
    top = np.floor(np.log2(masks)).astype(int)
    eps = np.finfo(np.float32).eps
    classes = [masks[top < 2 * n - 4]] + [masks[top == b] for b in range(2 * n - 4, 2 * n)]
    classes = [own for own in classes if own.size]        # Bravyi-Kitaev leaves one of the four empty
    assert len(classes) >= 4
    for own in classes:                                   # below the four classes, then each of them
        # the masks with the most bits among the four highest, and some others
        high = np.bitwise_count(own >> (2 * n - 4))
        pick = np.concatenate([own[np.argsort(-high, kind="stable")[:2]], rng.choice(own, 4)])
        for m in pick:
            cols = rng.integers(0, 1 << (2 * n), size=512)
            v = value_at(x, z, c, m, cols)
            col, v = int(cols[np.argmax(np.abs(v))]), float(v[np.argmax(np.abs(v))])
            got = []
            for s in (1.0, -1.0):
                psi = np.zeros(1 << (2 * n), complex)
                psi[col], psi[col ^ int(m)] = 1.0, s
                psi /= np.sqrt(2.0)
                st = to_state(ctx, psi, 2 * n, tq.TQ_C64)
                E = tq.energy(ctx, h64, st)
                ref = tq.energy(ctx, h128, to_state(ctx, st.numpy(), 2 * n, tq.TQ_C128))
                # one product per row, of a value rounded to float32; the diagonal is float64
                assert abs(E - ref) <= 2 * eps * abs(v) + 1e-12 * abs(ref)
                got.append(E)
            # the sides of the coupling, both: a lost or single count is off by |v|
            assert abs(v) > 1e-6
            assert abs(0.5 * (got[0] - got[1]) - v) <= 4 * eps * abs(v) + 1e-11


def test_rounding_no_larger_than_the_full_pass():
    q, ne, count = 16, 8, 48
    ctx = tq.Context(0)
    ints = synth.integrals(q // 2, 90)
    h64 = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, tq.TQ_JW, tq.TQ_C64)
    h128 = tq.build_hamiltonian(ctx, ints.h, ints.g, 0.0, tq.TQ_JW, tq.TQ_C128)
    pool = tq.build_pool(ctx, q // 2, ne, tq.TQ_JW)
    hf = torch.zeros(count, 1 << q, dtype=torch.complex128, device="cuda")
    hf[:, tq.hf_index(q, ne, tq.TQ_JW)] = 1.0
    gen = torch.Generator(device="cuda").manual_seed(4)
    for _ in range(60):
        k = torch.randint(0, pool.M, (count,), generator=gen, device="cuda", dtype=torch.int32)
        th = 0.4 * torch.randn(count, generator=gen, device="cuda", dtype=torch.float64)
        tq.evolve_taylor5_batch(ctx, pool, hf, k, th, prec=tq.TQ_C128)
    hf /= torch.linalg.norm(hf, dim=1, keepdim=True)
    err = []
    for sched in (None, 32):                              # the default, and the CSR with 32 sums a row
        if sched:
            ctx.set_spmv_schedule(sched)
        states = [hf[i].to(torch.complex64).contiguous() for i in range(count)]
        got = [tq.energy(ctx, h64, tq.State(ctx, q, tq.TQ_C64, tensor=s)) for s in states]
        ref = [tq.energy(ctx, h128, tq.State(ctx, q, tq.TQ_C128, tensor=s.to(torch.complex128))) for s in states]
        err.append(np.sqrt(np.mean(np.square(np.subtract(got, ref)))))
    # a root mean square over 48 states scatters by a tenth; the ratio of two
    # by a seventh: a quarter above one is far above it
    assert err[0] <= 1.25 * err[1]
