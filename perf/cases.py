"""The workloads this framework's speed is judged on, through its public entry
points.

Most of a user's time goes into sampling shots of a surface-code memory
(Simulator.sample_shots): many shots of a small code, one shot of it, a d = 5
code at the bond caps the threshold plots use, a d = 7 code with a few coupled
pairs.  Beside it stand the likelihood gradient that fits crosstalk angles and
the dense blocks of the truncation sweep (SVD, R factor, contraction), each
called alone, at the bond sizes a chi = 256 run reaches.  A whole chi = 256 run
takes minutes, so its large bonds appear here only as those blocks.
"""

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2605_29514_gb300 as stn

C128, C64 = 0, 1
CDTYPE = {C128: torch.complex128, C64: torch.complex64}
RDTYPE = {C128: torch.float64, C64: torch.float32}


def _shots(name, **kw):
    case = dict(name=name, kind="shots", distance=3, rounds=1, basis="Z", theta=0.05, p=1e-3, cap=32, precision=C64,
                shots=152, every=1, logical=False)
    case.update(kw)
    return case


def listed():
    return [
        # one shot of the exact d = 3 memory: interactive use, pure latency
        _shots("d3_one_shot_c128", precision=C128, p=0.0, cap=64, shots=1),
        # the exact d = 3 parity configuration: two rounds in complex128
        _shots("d3_exact_c128", precision=C128, p=0.0, cap=64, rounds=2, shots=100),
        # a point of a d = 3 logical-error curve: many shots, more than the GPU holds at once
        _shots("d3_curve_c64", shots=1000),
        # X-memory with the logical expectation before the readout (the angle behind the P_L estimator)
        _shots("d3_x_logical_c64", basis="X", theta=0.0225, shots=150, logical=True),
        # d = 5 at the crosstalk angle of the paper's device table
        _shots("d5_table_c64", distance=5, theta=1e-3),
        # d = 5, strong crosstalk, the bond cap of the threshold plots: the heaviest ordinary call
        _shots("d5_strong_c64", distance=5, theta=0.05),
        # d = 5 in complex128 with explicit pairs (one in four couplings), an odd number of shots
        _shots("d5_pairs_c128", distance=5, theta=0.0225, precision=C128, cap=16, shots=37, every=4),
        # d = 7 (two words per tableau row) with explicit pairs, a small cap
        _shots("d7_pairs_c64", distance=7, theta=0.0225, cap=8, shots=99, every=4),
        # one gradient of an angle fit on an X-memory: fixed records, d log P / d theta of a few pairs
        dict(name="d3_gradient_c128", kind="grad", theta=0.1, p=0.0, cap=64, records=48, every=3),
        # the truncation SVD of a large bond, from a caller that cannot allocate
        dict(name="svd_bond_c64", kind="svd", precision=C64, m=256, n=192),
        # the same in complex128 at the size where bonds leave shared memory
        dict(name="svd_bond_c128", kind="svd", precision=C128, m=72, n=66),
        # the R factor of the left sweep at a large bond
        dict(name="qr_bond_c64", kind="qr", precision=C64, m=512, n=250),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["d3", "d3", "d3x", "d5", "d7", "grad", "svd", "svd", "qr", "gemm"])
    theta = math.exp(rng.uniform(math.log(1e-3), math.log(0.05)))
    p = rng.choice([0.0, 1e-3, 5e-3])
    if kind == "d3":
        precision, rounds = rng.choice([C128, C64]), rng.choice([1, 1, 2])
        most = 300 if precision == C128 and rounds == 2 else 1000 if precision == C64 and rounds == 1 else 600
        return _without_name(_shots("", precision=precision, rounds=rounds, theta=theta, p=p, cap=64,
                                    shots=log_int(1, most), logical=rng.random() < 0.3))
    if kind == "d3x":
        theta = min(theta, 0.0225)
        return _without_name(_shots("", basis="X", theta=theta, p=p, shots=log_int(1, 152)))
    if kind == "d5":
        return _without_name(_shots("", distance=5, theta=theta, p=p, cap=rng.choice([5, 8, 12, 16, 32]),
                                    shots=log_int(1, 152), every=rng.choice([1, 2, 3])))
    if kind == "d7":
        return _without_name(_shots("", distance=7, theta=theta, p=p, cap=rng.choice([4, 7, 8]),
                                    shots=log_int(1, 152), every=rng.choice([4, 5, 6])))
    if kind == "grad":
        return dict(kind="grad", theta=theta * 2, p=p, cap=64, records=log_int(1, 64), every=rng.choice([3, 4, 5]))
    if kind == "svd":
        if rng.random() < 0.5:
            return dict(kind="svd", precision=C64, m=log_int(20, 400), n=log_int(20, 200))
        return dict(kind="svd", precision=C128, m=log_int(8, 128), n=log_int(8, 128))
    precision = rng.choice([C64, C64, C128])
    most = 512 if precision == C64 else 200
    if kind == "qr":
        return dict(kind="qr", precision=precision, m=log_int(8, most), n=log_int(4, most // 2))
    return dict(kind="gemm", precision=precision, op_a=rng.choice([0, 1]), op_b=rng.choice([0, 1]),
                m=log_int(4, most), n=log_int(4, most), k=log_int(4, most))


def _without_name(case):
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# inputs
def _pairs(case):
    """Every `every`-th coupled (ancilla, data) pair with the idle rule, or None for the default rule."""
    if case["every"] == 1:
        return None
    lay = _Layout(case["distance"])
    return tuple((a, q, "ZZ", None) for a, q in lay.couplings[:: case["every"]])


def _workload(case):
    cutoff = 1e-12 if case["precision"] == C128 else 5e-6
    return SimpleNamespace(distance=case["distance"], rounds=case["rounds"], pair_rule="adjacent_idle",
                           chi_cap=case["cap"], p=case["p"], p1_scale=0.1, p2_scale=1.0, pR_scale=2.0, pM_scale=5.0,
                           svd_cutoff=cutoff, degeneracy_tol=cutoff, precision=case["precision"], seed=0,
                           memory_basis=case["basis"], cnot_schedule=None, pairs=_pairs(case))


def _grad_case(case):
    return _shots("", precision=C128, basis="X", theta=case["theta"], p=case["p"], cap=case["cap"],
                  shots=case["records"], every=case["every"])


def _inputs(case, seed, n_pairs):
    """Quenched per-pair angles and the first global shot index."""
    rng = np.random.default_rng(seed)
    theta = rng.normal(case["theta"], 0.1 * case["theta"], size=n_pairs)
    return theta, int(rng.integers(0, 1 << 40))


def _unitary(g, m, n):
    """m x n with orthonormal columns."""
    a = torch.randn(m, n, 2, dtype=torch.float64, device="cuda", generator=g)
    return torch.linalg.qr(torch.view_as_complex(a))[0]


def _matrices(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    m, n = case["m"], case["n"]
    if case["kind"] == "gemm":
        k = case["k"]
        shapes = [(k, m) if case["op_a"] else (m, k), (n, k) if case["op_b"] else (k, n)]
        return [torch.randn(*s, dtype=CDTYPE[case["precision"]], device="cuda", generator=g) for s in shapes]
    # Schmidt values of a bond fall over six decades
    k = min(m, n)
    s = torch.exp(torch.arange(k, dtype=torch.float64, device="cuda") * (-math.log(1e6) / k))
    a = (_unitary(g, m, k) * s) @ _unitary(g, n, k).mH
    return [a.to(CDTYPE[case["precision"]]).contiguous()]


def prepare(case, seed):
    if case["kind"] in ("svd", "qr", "gemm"):
        return dict(case=case, mats=_matrices(case, seed), status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    sim_case = _grad_case(case) if case["kind"] == "grad" else case
    sim = stn.Simulator(_workload(sim_case), max_shots=sim_case["shots"],
                        stream=torch.cuda.current_stream().cuda_stream)
    theta, offset = _inputs(sim_case, seed, sim.n_pairs)
    state = dict(case=case, sim=sim, theta=theta, offset=offset)
    if case["kind"] == "grad":  # the measured records, at a slightly different angle
        state["records"] = sim.sample_shots(case["records"], offset, theta * 1.1, stats=False)["records"]
    return state


# ---------------------------------------------------------------------------
# one pass
def run(state):
    case = state["case"]
    if case["kind"] == "shots":
        sim, shots = state["sim"], case["shots"]
        logical = None
        if case["logical"]:
            sim.begin_batch(shots, state["offset"])
            for r in range(case["rounds"]):
                sim.apply_round(r, state["theta"])
            logical = sim.logical_expectation()
            sim.apply_round(case["rounds"], state["theta"])
            out = sim.read_records(stats=False)
        else:
            out = sim.sample_shots(shots, state["offset"], state["theta"], stats=False)
        # the type of the state the probabilities are norms of
        real = np.float64 if case["precision"] == C128 else np.float32
        got = {"records": out["records"], "born": out["born"].astype(real)}
        if logical is not None:
            got["logical"] = logical.astype(real)
        return got
    if case["kind"] == "grad":
        logp, grad = state["sim"].logprob_grad(state["records"], state["theta"], shot_offset=state["offset"])
        return {"logp": logp, "grad": grad}
    stream = torch.cuda.current_stream().cuda_stream
    precision, a = case["precision"], state["mats"][0]
    m, n = case["m"], case["n"]
    if case["kind"] == "qr":
        r = a.clone()
        stn.dense_qr(precision, m, n, r.data_ptr(), stream=stream)
        return r
    if case["kind"] == "gemm":
        b = state["mats"][1]
        c = torch.empty(m, n, dtype=a.dtype, device="cuda")
        stn.dense_cgemm(precision, case["op_a"], case["op_b"], m, n, case["k"], a.data_ptr(), a.shape[1], b.data_ptr(),
                        b.shape[1], c.data_ptr(), n, state["status"].data_ptr(), stream=stream)
        return c
    v = torch.empty(n, n, dtype=a.dtype, device="cuda")
    sig2 = torch.empty(n, dtype=RDTYPE[precision], device="cuda")
    stn.dense_svd_noalloc(precision, m, n, a.data_ptr(), v.data_ptr(), sig2.data_ptr(), stream=stream)
    # the truncation the decomposition is for: the singular values, largest first, and the matrix the largest keep
    sig2, order = torch.sort(sig2, descending=True)
    vk = v[order[: _keep(case)]]
    return {"sigma": sig2.sqrt(), "truncated": (a @ vk.mT) @ vk.conj()}


def _keep(case):
    return max(1, min(case["m"], case["n"]) * 3 // 4)


def work(case):
    """Floating-point operations: the textbook counts of the contractions, R factors and SVDs; for a simulation the
    framework's own count of them over the bonds the batch reaches, twice that for a gradient (there and back)."""
    if case["kind"] in ("shots", "grad"):
        c = _grad_case(case) if case["kind"] == "grad" else case
        st = prepare({**c, "logical": False}, 0)
        run(st)
        sim = st["sim"]
        flops = sim.algorithmic_flops() * (2 if case["kind"] == "grad" else 1)
        nbytes = 8 * sim.n_pairs + c["shots"] * (sim.rec_bytes + 8 * sim.n_meas)
        return {"bytes": nbytes, "flops": flops}
    elem = 16 if case["precision"] == C128 else 8
    m, n = case["m"], case["n"]
    hi, lo = max(m, n), min(m, n)
    if case["kind"] == "gemm":
        k = case["k"]
        return {"bytes": elem * (m * k + k * n + m * n), "flops": 8 * m * n * k}
    if case["kind"] == "qr":
        return {"bytes": 2 * elem * m * n, "flops": 4 * (2 * hi * lo * lo - 2 * lo ** 3 / 3)}
    return {"bytes": elem * (2 * m * n + n * n), "flops": 4 * (4 * hi * lo * lo + 8 * lo ** 3) + 16 * m * n * _keep(case)}


# ---------------------------------------------------------------------------
# the same in 64 bits with plain numpy and torch
class _Layout:
    """Rotated surface code: qubits in row-major order, CNOT layers, coupled pairs."""

    def __init__(self, d):
        pts = [(2 * j + 1, 2 * i + 1, "D") for j in range(d) for i in range(d)]
        for j in range(d + 1):
            for i in range(d + 1):
                kind = "X" if (i + j) % 2 else "Z"
                inner_i, inner_j = 1 <= i <= d - 1, 1 <= j <= d - 1
                if (inner_i and inner_j) or (inner_i and kind == "X" and j in (0, d)) or (
                        inner_j and kind == "Z" and i in (0, d)):
                    pts.append((2 * j, 2 * i, kind))
        pts.sort()
        self.n = len(pts)
        self.kind = [k for _, _, k in pts]
        self.xy = [(x, y) for y, x, _ in pts]
        at = {c: q for q, c in enumerate(self.xy)}
        self.data = [q for q in range(self.n) if self.kind[q] == "D"]
        self.anc = [q for q in range(self.n) if self.kind[q] != "D"]
        order = {"Z": [(-1, -1), (-1, 1), (1, -1), (1, 1)], "X": [(-1, -1), (1, -1), (-1, 1), (1, 1)]}
        self.slots = {a: [at.get((self.xy[a][0] + dx, self.xy[a][1] + dy)) for dx, dy in order[self.kind[a]]]
                      for a in self.anc}
        self.couplings = [(a, q) for a in self.anc for q in self.slots[a] if q is not None]


def _uniforms(shots, offset, events):
    """Philox4x32-10 with key 0 and counter (shot, event): doubles [shots][events]."""
    u = np.uint64
    mask = u(0xFFFFFFFF)
    s = (np.arange(shots, dtype=np.uint64) + u(offset))[:, None]
    c0, c1 = np.broadcast_arrays(s & mask, s >> u(32))
    c2 = np.arange(events, dtype=np.uint64)[None, :] + np.zeros_like(c0)
    c0, c1 = c0 + np.zeros_like(c2), c1 + np.zeros_like(c2)
    c3 = np.zeros_like(c2)
    k0 = k1 = 0
    for _ in range(10):
        a, b = u(0xD2511F53) * c0, u(0xCD9E8D57) * c2
        c0, c1, c2, c3 = (b >> u(32)) ^ c1 ^ u(k0), b & mask, (a >> u(32)) ^ c3 ^ u(k1), a & mask
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return ((c0 << u(21)) ^ (c1 >> u(11))).astype(np.float64) * 2.0 ** -53


class _Dense:
    """Dense amplitudes of a batch, [batch][tangent][2^n]: tangent 0 is the state, 1 + k its derivative by angle k."""

    def __init__(self, n, batch, tangents):
        self.n = n
        self.psi = torch.zeros(batch, tangents, 2 ** n, dtype=torch.complex128, device="cuda")
        self.psi[:, 0, 0] = 1

    def view(self, q, psi=None):
        psi = self.psi if psi is None else psi
        return psi.view(psi.shape[0], psi.shape[1], 2 ** q, 2, -1)

    def h(self, q):
        v = self.view(q)
        a, b = v[:, :, :, 0].clone(), v[:, :, :, 1].clone()
        v[:, :, :, 0] = (a + b) * math.sqrt(0.5)
        v[:, :, :, 1] = (a - b) * math.sqrt(0.5)

    def two(self, a, b):
        """View with the axes of qubits a and b at positions 3 and 5 (a at 3 when a < b)."""
        lo, hi = min(a, b), max(a, b)
        return self.psi.view(self.psi.shape[0], self.psi.shape[1], 2 ** lo, 2, 2 ** (hi - lo - 1), 2, -1)

    def cnot(self, c, t):
        v = self.two(c, t)
        if c < t:
            v[:, :, :, 1] = v[:, :, :, 1].flip(4)
        else:
            v[:, :, :, :, :, 1] = v[:, :, :, :, :, 1].flip(3)

    def paulis(self, q, letters):
        """letters[batch]: 0 I, 1 X, 2 Y, 3 Z (a global phase is left out)."""
        for s in np.nonzero((letters == 1) | (letters == 2))[0]:
            v = self.view(q)[s]
            v.copy_(v.flip(2))
        for s in np.nonzero((letters == 3) | (letters == 2))[0]:
            self.view(q)[s][:, :, 1] *= -1

    def rotate(self, a, b, theta, k):
        v = self.two(a, b)
        sign = torch.tensor([1.0, -1.0], dtype=torch.float64, device="cuda")
        zz = sign[:, None, None, None] * sign[None, None, :, None]
        v *= torch.exp(-1j * theta * zz)
        if k is not None and self.psi.shape[1] > 1:  # d/dtheta_k adds -i ZZ of the rotated state
            v[:, 1 + k] += -1j * zz * v[:, 0]

    def p0(self, q):
        v = self.view(q)[:, 0]
        w = v.real.square().sum(dim=(1, 3)) + v.imag.square().sum(dim=(1, 3))
        return (w[:, 0] / w.sum(dim=1)).cpu().numpy()

    def project(self, q, bits, norm):
        keep = torch.zeros(len(bits), 1, 1, 2, 1, dtype=torch.float64, device="cuda")
        keep[torch.arange(len(bits)), 0, 0, torch.from_numpy(bits.astype(np.int64)), 0] = torch.from_numpy(norm).cuda()
        v = self.view(q)
        v *= keep


def _dense_run(case, theta, offset, forced=None):
    """Records, Born probabilities and the logical expectation of a d = 3 batch; with forced records, log P and its
    gradient instead."""
    lay = _Layout(case["distance"])
    d, n, shots, p = case["distance"], lay.n, case["shots"], case["p"]
    x_memory = case["basis"] == "X"
    pairs = lay.couplings[:: case["every"]]
    idle = {pair: [layer for layer in range(4) if lay.slots[pair[0]][layer] != pair[1]] for pair in pairs}
    n_meas = case["rounds"] * len(lay.anc) + len(lay.data)
    u = _uniforms(shots, offset, 4096)
    st = _Dense(n, shots, 1 if forced is None else 1 + len(pairs))
    bits = np.zeros((shots, n_meas), dtype=np.uint8)
    born = np.zeros((shots, n_meas))
    ev, rec = 0, 0

    def flips(prob):
        nonlocal ev
        ev += 1
        return u[:, ev - 1] < prob

    def noise1(q):
        nonlocal ev
        x = u[:, ev]
        ev += 1
        p1 = 0.1 * p
        if p1 > 0:
            st.paulis(q, np.where(x < p1, 1 + np.minimum(2, (3 * x / p1).astype(int)), 0))

    def noise2(a, b):
        nonlocal ev
        x = u[:, ev]
        ev += 1
        if p > 0:
            idx = np.where(x < p, np.minimum(14, (15 * np.minimum(x / p, 1.0)).astype(int)) + 1, 0)
            st.paulis(a, idx // 4)
            st.paulis(b, idx % 4)

    def measure(q, reset):
        nonlocal ev, rec
        p0 = np.clip(st.p0(q), 0.0, 1.0)
        flip = u[:, ev + 1] < 5.0 * p
        bit = (u[:, ev] >= p0).astype(np.uint8)
        if forced is not None:
            bit = forced[:, rec] ^ flip
        pb = np.where(bit == 0, p0, 1.0 - p0)
        st.project(q, bit, np.ones(shots) if forced is not None else 1.0 / np.sqrt(pb))
        born[:, rec] = pb
        bits[:, rec] = bit ^ flip
        rec += 1
        ev += 2
        if reset:
            st.paulis(q, bit.astype(int))
            st.paulis(q, flips(2.0 * p).astype(int))

    for q in range(n):
        st.paulis(q, flips(2.0 * p).astype(int))
    if x_memory:
        for q in lay.data:
            st.h(q)
            noise1(q)
    x_anc = [a for a in lay.anc if lay.kind[a] == "X"]
    for _ in range(case["rounds"]):
        for a in x_anc:
            st.h(a)
            noise1(a)
        for layer in range(4):
            for a in lay.anc:
                q = lay.slots[a][layer]
                if q is not None:
                    c, t = (a, q) if lay.kind[a] == "X" else (q, a)
                    st.cnot(c, t)
                    noise2(c, t)
            for k, pair in enumerate(pairs):
                if layer in idle[pair]:
                    st.rotate(pair[0], pair[1], float(theta[k]), k)
        for a in x_anc:
            st.h(a)
            noise1(a)
        for a in lay.anc:
            measure(a, True)
    logical = None
    if case["logical"]:
        phi = st.psi.clone()
        for q in lay.data:
            if x_memory and lay.xy[q][0] == 1:
                v = st.view(q, phi)
                phi = v.flip(3).reshape(phi.shape)
            elif not x_memory and lay.xy[q][1] == 1:
                st.view(q, phi)[:, :, :, 1] *= -1
        logical = (st.psi.conj() * phi).sum(dim=(1, 2)).real.cpu().numpy()
        del phi
    if x_memory:
        for q in lay.data:
            st.h(q)
            noise1(q)
    for q in lay.data:
        measure(q, False)
    if forced is None:
        return np.packbits(bits, axis=1, bitorder="little"), born, logical
    inner = torch.einsum("bi,bki->bk", st.psi[:, 0].conj(), st.psi).cpu().numpy()
    return np.log(inner[:, 0].real), (2 * inner[:, 1:].real / inner[:, :1].real).sum(axis=0)


def _householder_r(a):
    """R of the Householder reflections that map each column x to -x_0 / |x_0| ||x|| e_1."""
    r = a.to(torch.complex128).clone()
    m, n = r.shape
    for j in range(min(m, n)):
        x = r[j:, j].clone()
        norm = torch.linalg.vector_norm(x)
        phase = torch.where(x[0].abs() > 0, x[0] / x[0].abs(), torch.ones_like(x[0]))
        x[0] += phase * norm
        w = x / torch.linalg.vector_norm(x)
        r[j:, j:] -= 2 * torch.outer(w, w.conj() @ r[j:, j:])
        r[j, j] = -phase * norm
        r[j + 1:, j] = 0
    return r


def exact(case, seed):
    if case["kind"] == "shots":
        if case["distance"] != 3:
            return None  # 49 and more qubits: no dense state
        theta, offset = _inputs(case, seed, len(_Layout(3).couplings[:: case["every"]]))
        parts = []
        for s in range(0, case["shots"], 256):
            part = {**case, "shots": min(256, case["shots"] - s)}
            parts.append(_dense_run(part, theta, offset + s))
        got = {"records": np.concatenate([x[0] for x in parts]), "born": np.concatenate([x[1] for x in parts])}
        if case["logical"]:
            got["logical"] = np.concatenate([x[2] for x in parts])
        return got
    if case["kind"] == "grad":
        sim_case = _grad_case(case)
        lay = _Layout(3)
        theta, offset = _inputs(sim_case, seed, len(lay.couplings[:: case["every"]]))
        records = _dense_run(sim_case, theta * 1.1, offset)[0]
        n_meas = len(lay.anc) + len(lay.data)
        forced = np.unpackbits(records, axis=1, bitorder="little")[:, :n_meas]
        logp, grad = [], 0.0
        for s in range(0, case["records"], 16):
            part = {**sim_case, "shots": min(16, case["records"] - s)}
            lp, g = _dense_run(part, theta, offset + s, forced[s: s + 16])
            logp.append(lp)
            grad = grad + g
        return {"logp": np.concatenate(logp), "grad": grad}
    mats = [x.to(torch.complex128) for x in _matrices(case, seed)]
    if case["kind"] == "qr":
        return _householder_r(mats[0])
    if case["kind"] == "gemm":
        a, b = mats
        return (a.mH if case["op_a"] else a) @ (b.mH if case["op_b"] else b)
    u, s, vh = torch.linalg.svd(mats[0], full_matrices=False)
    sigma = torch.zeros(case["n"], dtype=torch.float64, device="cuda")
    sigma[: len(s)] = s
    k = _keep(case)
    return {"sigma": sigma, "truncated": (u[:, :k] * s[:k]) @ vh[:k]}
