"""Timed cases of the ADAPT-VQE Taylor-5 framework, through its public Python entry points.

Every kind of call a program of this framework makes: one state update, the batched update, the
energy, all pool gradients, the adjoint gradient of an ansatz, ADAPT runs, many trajectories at once,
the Hamiltonian build and the request loop.  Molecules are seeded shape-matched integrals (h with a
sorted diagonal in [-2, 1] and small off-diagonals, g a sum of six symmetric factors), states are
Hartree-Fock followed by random pool rotations, as an ADAPT run leaves them.

``exact`` restates each call in 64 bits in the occupation-number basis: ladder operators with their
sign strings, the Hamiltonian as one value vector per index mask, and the Taylor series of a pool
generator A (A^3 = -A) in closed form.
"""

import ctypes
import math
import random

import numpy as np
import torch

import paper_2606_29692_gb300 as tq

JW, BK = tq.TQ_JW, tq.TQ_BK
PREC = {"c128": tq.TQ_C128, "c64": tq.TQ_C64}
DTYPE = {"c128": torch.complex128, "c64": torch.complex64}
BYTES = {"c128": 16, "c64": 8}
MAP = {"jw": JW, "bk": BK}
EPS = 1e-3

_ctx = None


def context():
    """One context for the process, as a program holds it."""
    global _ctx
    if _ctx is None:
        _ctx = tq.Context(0)
    return _ctx


# ------------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest call: one renormalised double-precision update of an 8-qubit state, the inner
        # step of a plain run on a small active space
        {"name": "update_8q_c128", "kind": "update", "qubits": 8, "electrons": 4, "map": "jw", "prec": "c128"},
        # one update of a state too large for one thread-block cluster
        {"name": "update_20q_c64", "kind": "update", "qubits": 20, "electrons": 10, "map": "bk", "prec": "c64"},
        # the headline: 8192 14-qubit states in place, each with its own generator and angle, in the
        # index layout the framework's planner gives for the pool
        {"name": "batch_14q_c64", "kind": "batch", "qubits": 14, "electrons": 6, "map": "bk", "prec": "c64",
         "states": 8192, "packed": True},
        # the energy of a 12-qubit, 8-electron molecule in double precision: a small call whose result
        # the host waits for
        {"name": "energy_12q_c128", "kind": "energy", "qubits": 12, "electrons": 8, "map": "jw", "prec": "c128"},
        # the energy of the largest served size
        {"name": "energy_18q_c64", "kind": "energy", "qubits": 18, "electrons": 8, "map": "bk", "prec": "c64"},
        # screening the whole pool at 14 qubits (strongly correlated integrals), result on the host
        {"name": "gradients_14q_c64", "kind": "gradients", "qubits": 14, "electrons": 6, "map": "bk", "prec": "c64",
         "strong": True, "host": True},
        # the same at 16 qubits in double precision, result left on the device
        {"name": "gradients_16q_c128", "kind": "gradients", "qubits": 16, "electrons": 8, "map": "jw",
         "prec": "c128", "strong": False, "host": False},
        # energy and gradient of a 20-factor ansatz (forward and adjoint sweep): what an optimiser of
        # all angles evaluates
        {"name": "ansatz_14q_c64", "kind": "ansatz", "qubits": 14, "electrons": 6, "map": "bk", "prec": "c64",
         "ops": 20},
        # a whole ADAPT run from Hartree-Fock with the line search: 12 qubits, 20 iterations
        {"name": "adapt_12q_c128", "kind": "adapt", "qubits": 12, "electrons": 8, "map": "jw", "prec": "c128",
         "iters": 20},
        # independent ADAPT trajectories of uneven size and length advanced together
        {"name": "trajectories_24_c64", "kind": "trajectories", "count": 24, "min_qubits": 10, "max_qubits": 14,
         "max_len": 30, "prec": "c64"},
        # building a 16-qubit Hamiltonian from integrals: once for every geometry of a scan
        {"name": "build_16q_c64", "kind": "build", "qubits": 16, "map": "bk", "prec": "c64"},
        # a burst of mixed requests (half updates, 30 % energies, 20 % gradients) on resident sessions
        {"name": "serve_96_c64", "kind": "serve", "requests": 96, "min_qubits": 12, "max_qubits": 16,
         "sessions": 24, "prec": "c64"},
    ]


def draw(rng):
    kind = rng.choice(["update", "batch", "energy", "gradients", "ansatz", "adapt", "trajectories", "build", "serve"])
    prec = rng.choice(["c64", "c128"])
    mp = rng.choice(["jw", "bk"])
    c = {"kind": kind, "prec": prec}
    if kind == "trajectories":
        c.update(count=rng.randint(3, 24), min_qubits=rng.choice([8, 10]), max_qubits=rng.choice([12, 14]),
                 max_len=rng.randint(5, 30))
    elif kind == "serve":
        c.update(requests=rng.randint(8, 96), min_qubits=rng.choice([8, 10, 12]), max_qubits=rng.choice([14, 16]),
                 sessions=rng.randint(4, 24))
    else:
        top = {"update": 22 if prec == "c64" else 20, "batch": 16, "energy": 18 if prec == "c64" else 16,
               "gradients": 18 if prec == "c64" else 16, "ansatz": 16, "adapt": 14, "build": 16}[kind]
        q = 2 * rng.randint(4, top // 2)
        c.update(qubits=q, map=mp)
        if kind != "build":
            c["electrons"] = rng.randint(2, min(q - 2, 10))
        if kind == "batch":
            most = 8192 * (1 << 14) * 8 // ((1 << q) * BYTES[prec])
            c.update(states=int(math.exp(rng.uniform(0.0, math.log(min(most, 20000))))), packed=rng.random() < 0.5)
        elif kind == "gradients":
            c.update(strong=rng.random() < 0.3 and c["electrons"] % 2 == 0, host=rng.random() < 0.5)
        elif kind == "ansatz":
            c["ops"] = rng.randint(1, 40)
        elif kind == "adapt":
            c["iters"] = rng.randint(2, 20)
    return c


# ------------------------------------------------------------------- inputs

def integrals(n, seed, strong=False, electrons=None):
    """Symmetric h and eightfold-symmetric g in chemist notation."""
    rng = np.random.default_rng(seed)
    h = np.diag(np.sort(rng.uniform(-2.0, 1.0, n)))
    o = np.triu(rng.normal(0.0, 0.05, (n, n)), 1)
    L = np.triu(rng.normal(0.0, 0.1, (6, n, n)))
    L = L + np.transpose(np.triu(L, 1), (0, 2, 1))
    if strong:
        o, L = 2.0 * o, 3.0 * L
        homo, lumo = electrons // 2 - 1, electrons // 2
        if 0 <= homo and lumo < n:
            h[lumo, lumo] = h[homo, homo] + 1e-3
    return h + o + o.T, np.einsum("lpq,lrs->pqrs", L, L)


def parity(v):
    for s in (16, 8, 4, 2, 1):
        v = v ^ (v >> s)
    return v & 1


def encode(occ, qubits, mapping, rows=None):
    """Basis index of each occupation bit string: JW is the string itself, BK the Fenwick-tree parities;
    ``rows`` then carries the index by a GF(2) map."""
    idx = occ
    if mapping == BK:
        idx = torch.zeros_like(occ)
        for k in range(qubits):
            low = (k + 1) & -(k + 1)
            mask = ((1 << (k + 1)) - 1) & ~((1 << (k + 1 - low)) - 1)
            idx |= parity(occ & mask) << k
    if rows is not None:
        out = torch.zeros_like(idx)
        for i, r in enumerate(rows):
            out |= parity(idx & int(r)) << i
        idx = out
    return idx


def excitations(n, electrons):
    """Spin-conserving singles, then doubles, from the lowest spin orbitals, each list lexicographic."""
    occ, vir = range(electrons), range(electrons, 2 * n)
    one = [(i, a) for i in occ for a in vir if i % 2 == a % 2]
    two = [(i, j, a, b) for i in occ for j in occ if j > i for a in vir for b in vir
           if b > a and i % 2 + j % 2 == a % 2 + b % 2]
    return one + two


def string(create, destroy):
    """(need1, need0, sign mask, sign) of create[0]^ create[1]^ .. destroy[0] destroy[1] .. on a ket:
    it acts on kets with need1 occupied and need0 empty, with sign (-1)^parity(ket & mask) * sign."""
    flipped, mask, sign = 0, 0, 1
    for p in reversed(list(create) + list(destroy)):
        below = (1 << p) - 1
        mask ^= below
        if bin(flipped & below).count("1") & 1:
            sign = -sign
        flipped ^= 1 << p
    need1 = sum(1 << p for p in destroy)
    return need1, sum(1 << p for p in create) & ~need1, mask, sign


class Generator:
    """A pool generator in the occupation basis: (A psi)[r] = a[r] psi[r ^ x]."""

    def __init__(self, exc, occ):
        half = len(exc) // 2
        one, zero, mask, sign = string(exc[half:], exc[half - 1::-1])

        def tau(ket):
            ok = ((ket & one) == one) & ((ket & zero) == 0)
            return torch.where(ok, sign * (1 - 2 * parity(ket & mask)), torch.zeros_like(ket))

        self.x = sum(1 << p for p in exc)
        self.src = occ ^ self.x
        self.a = (tau(self.src) - tau(occ)).to(torch.float64)

    def apply(self, psi):
        return self.a.to(psi.dtype) * psi[..., self.src]

    def combine(self, psi, on, off):
        """psi off the support, ``on`` psi + ``off`` A psi on it."""
        m = self.a.abs()
        f = 1.0 + (on - 1.0) * m if not torch.is_tensor(on) else 1.0 + (on[:, None] - 1.0) * m
        s = off * self.a if not torch.is_tensor(off) else off[:, None] * self.a
        return f.to(psi.dtype) * psi + s.to(psi.dtype) * psi[..., self.src]

    def rotate(self, psi, theta):
        return self.combine(psi, math.cos(theta), math.sin(theta))

    def taylor5(self, psi, t):
        t2 = t * t
        return self.combine(psi, 1.0 - t2 / 2 + t2 * t2 / 24, t * (1.0 - t2 / 6 + t2 * t2 / 120))

    def taylor5_slope(self, psi, t):
        """d/dt of the series: c4 A psi - s4 psi on the support, 0 off it."""
        t2 = t * t
        m = self.a.abs()
        return ((1.0 - t2 / 2 + t2 * t2 / 24) * self.a * psi[..., self.src]
                - t * (1.0 - t2 / 6) * m * psi)


def occupations(qubits):
    return torch.arange(1 << qubits, dtype=torch.int64, device="cuda")


def occupation_state(qubits, electrons, seed, dtype, depth=12):
    """Hartree-Fock followed by ``depth`` random pool rotations, normalised, in the occupation basis."""
    rng = np.random.default_rng(seed + 77)
    occ, exc = occupations(qubits), excitations(qubits // 2, electrons)
    psi = torch.zeros(1 << qubits, dtype=torch.complex128, device="cuda")
    psi[(1 << electrons) - 1] = 1.0
    for _ in range(depth):
        psi = Generator(exc[rng.integers(len(exc))], occ).rotate(psi, rng.normal(0.0, 0.3))
    return (psi / torch.linalg.vector_norm(psi)).to(dtype)


def to_index(psi, where):
    out = torch.empty_like(psi)
    out[..., where] = psi
    return out


def layout(case):
    """(mapping id of the calls, GF(2) rows or None): the base encoding, or the planner's packed one."""
    base = MAP[case["map"]]
    if not case.get("packed"):
        return base, None
    rows = tq.pool_sector_basis(case["qubits"] // 2, case["electrons"], base)
    return tq.mapping_linear(base, rows), [int(r) for r in rows]


def batch_inputs(case, seed):
    """States (occupation basis, the case's type), generators and angles of the batched update."""
    q, ne, n = case["qubits"], case["electrons"], case["states"]
    rng = np.random.default_rng(seed + 3)
    exc, occ = excitations(q // 2, ne), occupations(q)
    psi = torch.zeros((n, 1 << q), dtype=DTYPE[case["prec"]], device="cuda")
    psi[:, (1 << ne) - 1] = 1.0
    for _ in range(3):
        each_generator(psi, exc, occ, rng.integers(len(exc), size=n), rng.normal(0.0, 0.1, n), "rotate")
    return psi, rng.integers(len(exc), size=n).astype(np.int32), rng.normal(0.0, 0.1, n)


def each_generator(psi, exc, occ, k, theta, what):
    """psi[b] <- rotation or Taylor-5 update with generator k[b] and angle theta[b], in place."""
    for g in np.unique(k):
        at = np.nonzero(k == g)[0]
        A = Generator(exc[g], occ)
        for part in np.array_split(at, -(-len(at) * psi.shape[1] // (1 << 26))):
            rows = torch.as_tensor(part, device="cuda")
            t = torch.as_tensor(theta[part], device="cuda")
            if what == "rotate":
                psi[rows] = A.combine(psi[rows], torch.cos(t), torch.sin(t))
            else:
                t2 = t * t
                psi[rows] = A.combine(psi[rows], 1.0 - t2 / 2 + t2 * t2 / 24, t * (1.0 - t2 / 6 + t2 * t2 / 120))


def molecule(case, seed):
    return integrals(case["qubits"] // 2, seed, case.get("strong", False), case.get("electrons"))


def trajectory_list(case, seed):
    """(qubits, electrons, mapping, angles, integral seed) of each trajectory: sizes and lengths are the
    case's, angles and integrals the seed's."""
    size, rng = np.random.default_rng(11), np.random.default_rng(seed + 11)
    out = []
    for i in range(case["count"]):
        q = 2 * int(size.integers(case["min_qubits"] // 2, case["max_qubits"] // 2 + 1))
        length = case["max_len"] if i == 0 else int(size.integers(1, case["max_len"] + 1))
        out.append((q, 2 * (q // 4), int(size.integers(0, 2)), rng.normal(0.0, 0.1, length), seed + 1000 + i))
    return out


def serve_plan(case, seed):
    """Molecules [(qubits, electrons, mapping, integral seed)], the molecule of each session, and the
    requests [(kind, session, op, theta)]."""
    rng = np.random.default_rng(seed + 4)
    sizes = range(case["min_qubits"], case["max_qubits"] + 1, 2)
    mols = [(q, 2 * (q // 4), j % 2, seed + 2000 + j) for j, q in enumerate(sizes)]
    sess = [i % len(mols) for i in range(case["sessions"])]
    reqs = []
    for _ in range(case["requests"]):
        s = int(rng.integers(len(sess)))
        q, ne = mols[sess[s]][:2]
        reqs.append((int(rng.choice(3, p=(0.5, 0.3, 0.2))), s, int(rng.integers(len(excitations(q // 2, ne)))),
                     float(rng.normal(0.0, 0.1))))
    return mols, sess, reqs


class Borrowed:
    """A tensor over device memory that a handle of the framework owns; the tensor keeps this object,
    and with it the owner, alive."""

    def __init__(self, owner, ptr, shape, kind):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": shape, "typestr": kind, "data": (int(ptr), False), "version": 3}

    def tensor(self):
        return torch.as_tensor(self, device="cuda")


def states_of(call, owner, count, prec):
    """The resident states of a batch or server as tensors."""
    out = []
    for i in range(count):
        ptr, nq = ctypes.c_void_p(), ctypes.c_int()
        if call(owner.handle, i, ctypes.byref(ptr), ctypes.byref(nq)) != 0:
            raise RuntimeError(tq.lib().tq_last_error().decode())
        out.append(Borrowed(owner, ptr.value, (1 << nq.value,), "<c16" if prec == "c128" else "<c8").tensor())
    return out


# ------------------------------------------------------------------- prepare and run

def prepare(case, seed):
    kind, prec = case["kind"], case["prec"]
    p = PREC[prec]
    s = {"case": case}
    if kind == "trajectories":
        ctx, tr = context(), trajectory_list(case, seed)
        hams, pools = [], []
        for q, ne, mp, _, sd in tr:
            hams.append(tq.build_hamiltonian(ctx, *integrals(q // 2, sd), mapping=mp, prec=p))
            pools.append(tq.build_pool(ctx, q // 2, ne, mp))
        s["batch"] = tq.Batch(ctx, hams, pools, [t[1] for t in tr], [t[2] for t in tr], [t[3] for t in tr], EPS)
        s["states"] = states_of(tq.lib().tq_batch_state, s["batch"], len(tr), prec)
        return s
    if kind == "serve":
        mols, sess, reqs = serve_plan(case, seed)
        ctx = tq.Context(0)              # the server owns its context
        srv = tq.Server(ctx, p, hbm_budget=1 << 30, max_batch=256)
        ids = []
        for q, ne, mp, sd in mols:
            ids.append(srv.add_hamiltonian(tq.build_hamiltonian(ctx, *integrals(q // 2, sd), mapping=mp, prec=p),
                                           tq.build_pool(ctx, q // 2, ne, mp)))
        for m in sess:
            srv.add_session(ids[m], mols[m][1], mols[m][2])
        s["states"] = states_of(tq.lib().tq_server_session_state, srv, len(sess), prec)
        srv.start()
        s.update(server=srv, requests=reqs)
        return s
    ctx, q = context(), case["qubits"]
    mapping, rows = layout(case) if kind == "batch" else (MAP[case["map"]], None)
    if kind == "build":
        s["h"], s["g"] = integrals(q // 2, seed)
        return s
    ne = case["electrons"]
    if kind != "energy":
        s["pool"] = tq.build_pool(ctx, q // 2, ne, mapping)
    if kind not in ("update", "batch"):
        s["ham"] = tq.build_hamiltonian(ctx, *molecule(case, seed), mapping=mapping, prec=p)
    where = encode(occupations(q), q, MAP[case["map"]], rows)
    rng = np.random.default_rng(seed + 5)
    if kind == "batch":
        psi, k, th = batch_inputs(case, seed)
        s["psi"] = to_index(psi, where)
        s["k"] = torch.as_tensor(k, device="cuda")
        s["theta"] = torch.as_tensor(th, device="cuda")
        s["norm2"] = torch.linalg.vector_norm(psi, dim=1, dtype=DTYPE["c128"]).square()
        return s
    if kind in ("update", "ansatz"):
        ops = rng.integers(s["pool"].M, size=case.get("ops", 1))
        s["ops"], s["thetas"] = [int(k) for k in ops], [float(t) for t in rng.normal(0.0, 0.1, len(ops))]
    if kind in ("ansatz", "adapt"):
        s["state"] = tq.State(ctx, q, p)
        tq.state_set_hf(s["state"], ne, mapping)
        if kind == "ansatz":
            s["out"] = tq.State(ctx, q, p)
        return s
    s["state"] = tq.State(ctx, q, p, tensor=to_index(occupation_state(q, ne, seed, DTYPE[prec]), where))
    if kind == "gradients" and not case["host"]:
        s["g"] = torch.zeros(s["pool"].M, dtype=torch.float64, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind, p = case["kind"], PREC[case["prec"]]
    if kind == "update":
        tq.evolve_taylor5(context(), s["pool"], s["ops"][0], s["thetas"][0], s["state"], renormalize=True)
        return s["state"].tensor
    if kind == "batch":
        tq.evolve_taylor5_batch_support(context(), s["pool"], s["psi"], s["k"], s["theta"], s["norm2"], prec=p)
        return {"psi": s["psi"], "norm2": s["norm2"]}
    if kind == "energy":
        return tq.energy(context(), s["ham"], s["state"])
    if kind == "gradients":
        return tq.pool_gradients(context(), s["ham"], s["pool"], s["state"], out=s.get("g"))
    if kind == "ansatz":
        e, g = tq.ansatz_energy_grad(context(), s["ham"], s["pool"], s["state"], s["ops"], s["thetas"],
                                     psi_out=s["out"])
        return {"energy": e, "grad": g, "psi": s["out"].tensor}
    if kind == "adapt":
        tq.state_set_hf(s["state"], case["electrons"], MAP[case["map"]])
        steps, done = tq.adapt_run(context(), s["ham"], s["pool"], s["state"], EPS, case["iters"])
        out = {k: np.array([r[k] for r in steps]) for k in ("energy", "max_grad", "theta", "selected")}
        out.update(done=done, psi=s["state"].tensor)
        return out
    if kind == "trajectories":
        s["batch"].run()
        res = s["batch"].results()
        out = {k: np.concatenate([np.pad(r[k], (0, case["max_len"] - r["n_iter"])) for r in res])
               for k in ("energy", "max_grad", "theta", "selected")}
        out.update(n_iter=np.array([r["n_iter"] for r in res]), psi=s["states"])
        return out
    if kind == "build":
        ham = tq.build_hamiltonian(context(), s["h"], s["g"], mapping=MAP[case["map"]], prec=p)
        s["ham"] = ham                   # the last one built is kept, as a program keeps it
        d = 1 << case["qubits"]
        f = "<f8" if case["prec"] == "c128" else "<f4"
        rp, cl, vl, dg = tq.ham_csr(ham)
        nb, npairs, xp, xm, xv = tq.ham_xell(ham)
        arrays = {"rowptr": (rp, d + 1, "<i4"), "col": (cl, ham.nnz, "<i4"), "val": (vl, ham.nnz, f),
                  "diag": (dg, d, "<f8"), "xptr": (xp, nb + 1, "<i4"), "xmask": (xm, npairs, "<i4"),
                  "xval": (xv, 8 * npairs, f)}
        return {k: Borrowed(ham, ptr, (n,), t).tensor() for k, (ptr, n, t) in arrays.items()}
    srv, reqs = s["server"], s["requests"]
    for tag, (what, session, op, theta) in enumerate(reqs):
        srv.submit(what, session, op=op, theta=theta, tag=tag)
    got = []
    while len(got) < len(reqs):
        got += srv.poll(timeout_us=100000)
    got.sort(key=lambda c: c["tag"])
    out = {k: np.array([c[k] for c in got]) for k in ("energy", "max_grad", "norm2", "argmax", "status")}
    out["psi"] = s["states"]
    return out


# ------------------------------------------------------------------- work

def entries(qubits):
    """Off-diagonal non-zeros of a molecular Hamiltonian: singles and doubles of every determinant."""
    n, nnz = qubits // 2, 0
    for a in range(n + 1):
        for b in range(n + 1):
            sa, sb = a * (n - a), b * (n - b)
            pairs = math.comb(a, 2) * math.comb(n - a, 2) + math.comb(b, 2) * math.comb(n - b, 2)
            nnz += math.comb(n, a) * math.comb(n, b) * (sa + sb + sa * sb + pairs)
    return nnz


def h_bytes(qubits, prec):
    """The Hamiltonian once: diagonal, column and value of every entry."""
    return 8 * (1 << qubits) + (4 + BYTES[prec] // 2) * entries(qubits)


def pool_rows(qubits, electrons):
    """(pool size, support rows of the whole pool)."""
    exc, d = excitations(qubits // 2, electrons), 1 << qubits
    return len(exc), sum(d // 2 if len(e) == 2 else d // 8 for e in exc)


def work(case):
    kind, prec = case["kind"], case["prec"]
    if kind == "trajectories":
        # angles and lengths are drawn: half the longest length on average
        steps, b, f = (case["max_len"] + 1) / 2 * case["count"], 0.0, 0.0
        for q in range(case["min_qubits"], case["max_qubits"] + 1, 2):
            b += h_bytes(q, prec) + BYTES[prec] * 2 * (1 << q)
            f += 4.0 * entries(q) + 6.0 * pool_rows(q, 2 * (q // 4))[1]
        n = (case["max_qubits"] - case["min_qubits"]) // 2 + 1
        return {"bytes": steps * b / n, "flops": steps * f / n}
    if kind == "serve":
        sizes = list(range(case["min_qubits"], case["max_qubits"] + 1, 2))
        b = sum(0.5 * h_bytes(q, prec) + BYTES[prec] * 2 * (1 << q) for q in sizes) / len(sizes)
        f = sum(2.0 * entries(q) + 1.2 * pool_rows(q, 2 * (q // 4))[1] for q in sizes) / len(sizes)
        return {"bytes": case["requests"] * b, "flops": case["requests"] * f}
    q = case["qubits"]
    d, e = 1 << q, BYTES[prec]
    if kind == "update":
        return {"bytes": 2 * d * e, "flops": 10 * d}
    if kind == "build":
        pairs = entries(q) / 4.0            # about half of each pair's eight slots hold an entry
        return {"bytes": h_bytes(q, prec) + 4 * d + pairs * (4 + 4 * e), "flops": 8.0 * entries(q)}
    m, rows = pool_rows(q, case["electrons"])
    if kind == "batch":
        return {"bytes": case["states"] * (2.0 * rows / m * e + 28), "flops": case["states"] * 8.0 * rows / m}
    b, f = h_bytes(q, prec) + d * e, 4.0 * entries(q)
    if kind == "energy":
        return {"bytes": b, "flops": f}
    if kind == "gradients":
        return {"bytes": b + 8 * m, "flops": f + 6.0 * rows}
    if kind == "ansatz":
        return {"bytes": b + d * e + 8 * case["ops"], "flops": f + case["ops"] * 30.0 * rows / m}
    return {"bytes": case["iters"] * b, "flops": case["iters"] * (f + 6.0 * rows)}


# ------------------------------------------------------------------- exact

class Exact:
    """H and the pool of a molecule in 64 bits over the occupation basis."""

    def __init__(self, qubits, h, g):
        n, N = qubits // 2, qubits
        self.occ = occupations(qubits)
        terms = []
        for P in range(N):
            for Q in range(P % 2, N, 2):
                terms.append((h[P // 2, Q // 2], (P,), (Q,)))
        for P in range(N):
            for R in range(P + 1, N):
                for Q in range(N):
                    for S in range(Q + 1, N):
                        v = 0.0
                        if P % 2 == Q % 2 and R % 2 == S % 2:
                            v += g[P // 2, Q // 2, R // 2, S // 2]
                        if P % 2 == S % 2 and R % 2 == Q % 2:
                            v -= g[P // 2, S // 2, R // 2, Q // 2]
                        if v != 0.0:
                            terms.append((v, (P, R), (S, Q)))
        rec = []
        for v, cr, an in terms:
            x = 0
            for p in cr + an:
                x ^= 1 << p
            one, zero, mask, sign = string(cr, an)
            rec.append((x, one, zero, mask, v * sign))
        rec.sort(key=lambda r: r[0])
        self.x = sorted({r[0] for r in rec})
        at = {x: i for i, x in enumerate(self.x)}
        d = 1 << qubits
        # F[i, c] = H[c ^ x_i][c]; H is symmetric, so it is H[c][c ^ x_i] too
        self.F = torch.zeros((len(self.x), d), dtype=torch.float64, device="cuda")
        step = max(1, (1 << 23) // d)
        for i in range(0, len(rec), step):
            part = rec[i:i + step]
            col = lambda j, dt=torch.int64: torch.tensor([r[j] for r in part], dtype=dt, device="cuda")[:, None]  # noqa: E731
            ok = ((self.occ & col(1)) == col(1)) & ((self.occ & col(2)) == 0)
            val = (1 - 2 * parity(self.occ & col(3))).to(torch.float64) * col(4, torch.float64) * ok
            where = torch.tensor([at[r[0]] for r in part], device="cuda")
            self.F.index_add_(0, where, val)
        self.masks = torch.tensor(self.x, device="cuda")

    def apply(self, psi):
        w = torch.zeros_like(psi)
        step = max(1, (1 << 25) // psi.numel())
        for i in range(0, len(self.x), step):
            w += (self.F[i:i + step] * psi[self.occ ^ self.masks[i:i + step, None]]).sum(0)
        return w


def dot(a, b):
    return float(torch.vdot(a, b).real)


def exact_gradients(gens, psi, w, norm2):
    return np.array([2.0 * dot(w, A.apply(psi)) / norm2 for A in gens])


def exact_select(g, prec):
    a = np.abs(g)
    top = float(a.max())
    tau = 1e-9 * max(1.0, top) if prec == "c128" else 1e-5
    return int(np.nonzero(a >= top - tau)[0][0]), top


def exact_angle(H, A, psi, norm2):
    """The global minimiser of the energy along exp(theta A) psi: 4096 samples, ties to the smallest
    angle, then Newton steps."""
    u1 = A.apply(psi)
    u2 = A.apply(u1)
    w0, w1, w2 = H.apply(psi), H.apply(u1), H.apply(u2)
    h01, h02, h11, h12, h22 = (v / norm2 for v in (dot(w0, u1), dot(w0, u2), dot(w1, u1), dot(w1, u2), dot(w2, u2)))
    h00 = dot(w0, psi) / norm2

    def e(t):
        s, u = np.sin(t), 1.0 - np.cos(t)
        return h00 + 2 * s * h01 + 2 * u * h02 + s * s * h11 + 2 * s * u * h12 + u * u * h22

    step = 2.0 * math.pi / 4096
    t = -math.pi + step * (np.arange(4096) + 1)
    v = e(t)
    near = np.nonzero(v <= v.min() + 1e-10 * max(1.0, abs(v.min())))[0]
    t0 = th = float(t[near[np.argmin(np.abs(t[near]))]])
    for _ in range(8):
        s, c = math.sin(th), math.cos(th)
        u = 1.0 - c
        d1 = 2 * c * h01 + 2 * s * h02 + 2 * s * c * h11 + 2 * (c * u + s * s) * h12 + 2 * u * s * h22
        d2 = (-2 * s * h01 + 2 * c * h02 + 2 * (c * c - s * s) * h11 + 2 * (3 * s * c - s * u) * h12
              + 2 * (s * s + u * c) * h22)
        if not d2 > 0.0 or abs(th - d1 / d2 - t0) > step:
            break
        th -= d1 / d2
        if abs(d1 / d2) < 1e-15:
            break
    return t0 if e(th) > e(t0) else th


def exact_adapt(H, gens, psi, prec, steps, angles=None, renormalise=True):
    """[(energy, max|g|, angle, op)] of an ADAPT loop, and the state it ends with."""
    out = []
    for i in range(steps):
        norm2, w = dot(psi, psi), H.apply(psi)
        k, top = exact_select(exact_gradients(gens, psi, w, norm2), prec)
        if top < EPS:
            out.append((dot(psi, w) / norm2, top, 0.0, k))
            break
        t = exact_angle(H, gens[k], psi, norm2) if angles is None else float(angles[i])
        out.append((dot(psi, w) / norm2, top, t, k))
        psi = gens[k].taylor5(psi, t)
        if renormalise:
            psi = psi / torch.linalg.vector_norm(psi)
    return out, psi


def basis_state(qubits, electrons):
    psi = torch.zeros(1 << qubits, dtype=torch.complex128, device="cuda")
    psi[(1 << electrons) - 1] = 1.0
    return psi


def records(rec):
    out = {k: np.array(v, dtype=np.float64) for k, v in zip(("energy", "max_grad", "theta"), zip(*rec))}
    out["selected"] = None
    return out


def exact(case, seed):
    kind, prec = case["kind"], case["prec"]
    if kind == "trajectories":
        rec, states = [], []
        for q, ne, mp, angles, sd in trajectory_list(case, seed):
            H = Exact(q, *integrals(q // 2, sd))
            gens = [Generator(x, H.occ) for x in excitations(q // 2, ne)]
            r, psi = exact_adapt(H, gens, basis_state(q, ne), prec, len(angles), angles)
            rec += r + [(0.0, 0.0, 0.0, 0)] * (case["max_len"] - len(r))
            states.append(to_index(psi, encode(H.occ, q, mp)))
        return {**records(rec), "n_iter": None, "psi": states}
    if kind == "serve":
        mols, sess, reqs = serve_plan(case, seed)
        Hs = [Exact(q, *integrals(q // 2, sd)) for q, _, _, sd in mols]
        psis = [basis_state(*mols[m][:2]) for m in sess]
        out = {"energy": [], "max_grad": [], "norm2": []}
        for what, s, op, theta in reqs:
            (q, ne, _, _), H, psi = mols[sess[s]], Hs[sess[s]], psis[s]
            exc = excitations(q // 2, ne)
            e = top = 0.0
            norm2 = dot(psi, psi)
            if what == 0:
                psi = Generator(exc[op], H.occ).taylor5(psi, theta)
                norm2 = dot(psi, psi)
                psis[s] = psi / math.sqrt(norm2)
            else:
                w = H.apply(psi)
                e = dot(psi, w) / norm2
                if what == 2:
                    top = exact_select(exact_gradients((Generator(x, H.occ) for x in exc), psi, w, norm2), prec)[1]
            for k, v in (("energy", e), ("max_grad", top), ("norm2", norm2)):
                out[k].append(v)
        out = {k: np.array(v) for k, v in out.items()}
        out.update(argmax=None, status=None)
        out["psi"] = [to_index(psi, encode(occupations(mols[m][0]), mols[m][0], mols[m][2]))
                      for psi, m in zip(psis, sess)]
        return out
    q = case["qubits"]
    occ, base = occupations(q), MAP[case["map"]]
    if kind == "build":
        H = Exact(q, *integrals(q // 2, seed))
        where = encode(occ, q, base)
        masks = encode(H.masks, q, base)           # the encoding is linear over GF(2)
        order = torch.argsort(masks)
        order = order[masks[order] != 0]
        F = torch.empty((len(order), 1 << q), dtype=torch.float64, device="cuda")
        F[:, where] = H.F[order]
        diag = torch.empty(1 << q, dtype=torch.float64, device="cuda")
        diag[where] = H.F[H.x.index(0)]
        F[F.abs() <= 1e-11 * float(F.abs().max())] = 0.0
        keep = F.T != 0                            # rows, groups by ascending mask
        r, g = keep.nonzero(as_tuple=True)
        cols = r ^ masks[order][g]
        by = torch.argsort(r * (1 << q) + cols)
        blocks = F.reshape(len(order), -1, 8)
        b, gb = (blocks != 0).any(2).T.nonzero(as_tuple=True)
        return {"rowptr": None, "col": None, "val": F[g[by], r[by]], "diag": diag, "xptr": None, "xmask": None,
                "xval": blocks[gb, b].reshape(-1)}
    ne = case["electrons"]
    exc = excitations(q // 2, ne)
    where = encode(occ, q, base, layout(case)[1] if kind == "batch" else None)
    if kind == "batch":
        psi, k, th = batch_inputs(case, seed)
        psi = psi.to(torch.complex128)
        each_generator(psi, exc, occ, k, th, "taylor5")
        norm2 = torch.linalg.vector_norm(psi, dim=1).square()
        return {"psi": to_index(psi, where), "norm2": norm2}
    rng = np.random.default_rng(seed + 5)
    if kind in ("update", "ansatz"):
        ops = [int(k) for k in rng.integers(len(exc), size=case.get("ops", 1))]
        thetas = [float(t) for t in rng.normal(0.0, 0.1, len(ops))]
    if kind == "update":
        psi = occupation_state(q, ne, seed, DTYPE[prec]).to(torch.complex128)
        psi = Generator(exc[ops[0]], occ).taylor5(psi, thetas[0])
        return to_index(psi / torch.linalg.vector_norm(psi), where)
    H = Exact(q, *molecule(case, seed))
    if kind == "adapt":
        gens = [Generator(x, occ) for x in exc]
        rec, psi = exact_adapt(H, gens, basis_state(q, ne), prec, case["iters"])
        rec += rec[-1:] * (case["iters"] - len(rec))       # steps after convergence repeat it
        return {**records(rec), "done": None, "psi": to_index(psi, where)}
    if kind == "ansatz":
        gens = [Generator(exc[k], occ) for k in ops]
        phi = [basis_state(q, ne)]
        for A, t in zip(gens, thetas):
            phi.append(A.taylor5(phi[-1], t))
        norm2, w = dot(phi[-1], phi[-1]), H.apply(phi[-1])
        e = dot(phi[-1], w) / norm2
        chi, grad = w - e * phi[-1], np.zeros(len(ops))
        for j in range(len(ops) - 1, -1, -1):
            grad[j] = 2.0 * dot(chi, gens[j].taylor5_slope(phi[j], thetas[j])) / norm2
            chi = gens[j].taylor5(chi, -thetas[j])
        return {"energy": e, "grad": grad, "psi": to_index(phi[-1], where)}
    psi = occupation_state(q, ne, seed, DTYPE[prec]).to(torch.complex128)
    norm2, w = dot(psi, psi), H.apply(psi)
    if kind == "energy":
        return dot(psi, w) / norm2
    return exact_gradients((Generator(x, occ) for x in exc), psi, w, norm2)


if __name__ == "__main__":
    r = random.Random(0)
    for c in listed() + [draw(r) for _ in range(8)]:
        print(c, work(c))
