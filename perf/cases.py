"""The calls a user of this simulator makes, at the sizes they make them, for timing.

Every case compiles its circuit (or circuits) in `prepare`, as a program that simulates one
circuit keeps its handle, and makes one whole call in `run`: launch, tally, free. The circuits
are the package's own seeded workloads; `seed` keys the noise and outcome stream and the range
of shots, so another seed is another set of shots. Shots keep their records and status bytes
where a program would look at them (REC_ALL into its own device buffers), and only the
post-selection counters where it would not (the largest runs).
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2512_23037_gb300 as S
from paper_2512_23037_gb300 import circuits as C
from paper_2512_23037_gb300.grad import PostSelectedFidelity

TALLY = ("shots", "discarded", "overflow", "kept", "logical_errors")


def listed():
    return [
        # the smallest call: the 6-qubit workload, a few thousand shots, every record kept
        {"name": "tiny6_fp64", "kind": "shots", "circuit": "tiny6", "precision": "fp64", "n": 4096, "p": 1e-3,
         "records": True},
        # one point of a sweep over the noise rate: compile at that rate, run, read the tally
        {"name": "sweep_point", "kind": "sweep", "circuit": "w42", "precision": "fp32", "n": 262147, "p": 2e-3},
        # an ordinary run with records: the 42-qubit post-selected circuit, an odd million shots
        {"name": "w42_fp32_records", "kind": "shots", "circuit": "w42", "precision": "fp32", "n": 1000003, "p": 1e-3,
         "records": True},
        # the headline throughput run: 2^24 shots, post-selection counters only
        {"name": "w42_fp32_large", "kind": "shots", "circuit": "w42", "precision": "fp32", "n": 1 << 24, "p": 1e-3,
         "records": False},
        # the same circuit in the default precision
        {"name": "w42_fp64", "kind": "shots", "circuit": "w42", "precision": "fp64", "n": 1 << 22, "p": 1e-3,
         "records": True},
        # the large register: 97 qubits, maps of 64 entries and more, FP32 and FP64
        {"name": "w97_fp32", "kind": "shots", "circuit": "w97", "precision": "fp32", "n": 2000003, "p": 5e-4,
         "records": True},
        {"name": "w97_fp64", "kind": "shots", "circuit": "w97", "precision": "fp64", "n": 500009, "p": 5e-4,
         "records": True},
        # every op kind, no post-selection: outcomes are sampled all along, every shot runs to the end
        {"name": "random40_fp64", "kind": "shots", "circuit": "random40", "precision": "fp64", "n": 200003, "p": 1e-3,
         "records": True},
        # many circuits in one launch sequence (64 windowed circuits of 17-49 qubits)
        {"name": "batch64_fp32", "kind": "batch", "circuits": 64, "mean": 100000.0, "precision": "fp32", "set": 2},
        # the variance-reduced logical error rate: exact fidelity of the kept shots
        {"name": "fidelity_w42", "kind": "fidelity", "circuit": "w42", "precision": "fp32", "n": 2097169, "p": 1e-3},
        # post-selected fidelity and its gradient per error pattern, 72 angles
        {"name": "grad_w42rz_fp64", "kind": "grad", "precision": "fp64", "n": 100003},
        # one training step on a small parameterised circuit, through autograd
        {"name": "train_step_fp32", "kind": "train", "circuit_seed": 702, "qubits": 5, "ops": 94, "params": 6,
         "p": 0.02, "precision": "fp32", "n": 4099},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["shots", "shots", "shots", "window", "window", "sweep", "batch", "fidelity", "grad", "train"])
    prec = rng.choice(["fp32", "fp64"])
    if kind == "shots":
        name = rng.choice(["tiny6", "w42", "w42", "w97", "random40"])
        if name == "random40":  # sampled outcomes all along: the default precision
            prec = "fp64"
        top = {"tiny6": 1 << 20, "w42": 1 << (24 if prec == "fp32" else 22),
               "w97": 2000003 if prec == "fp32" else 500009, "random40": 200003}[name]
        p = _noise(rng, 3e-4, 1.2e-3) if name == "w97" else _noise(rng, 5e-4, 2e-3)
        n = _log(rng, 1024, top if p <= 1e-3 else top // 2)
        return {"kind": kind, "circuit": name, "precision": prec, "n": n, "p": p, "records": n <= 1 << 22}
    if kind == "window":  # other windowed circuits, of the ranges of the batch's
        w, blocks, p = rng.randint(2, 6), rng.randint(6, 24), _noise(rng, 1e-4, 3e-3)
        top = 3.0e6 / (1.0 + (4.0 ** w) / 100.0) * (1.0 if prec == "fp32" else 0.5)
        return {"kind": "shots", "circuit": "window", "w": w, "blocks": blocks, "qubits": rng.randint(17, 49),
                "circuit_seed": rng.randint(2000, 9999), "precision": prec, "n": _log(rng, 1024, top), "p": p,
                "records": rng.random() < 0.5}
    if kind == "sweep":
        return {"kind": kind, "circuit": rng.choice(["w42", "w42", "w97"]), "precision": prec,
                "n": _log(rng, 10000, 300000), "p": _noise(rng, 5e-4, 1e-3)}
    if kind == "batch":
        return {"kind": kind, "circuits": rng.randint(2, 64), "mean": float(_log(rng, 1000, 60000)), "precision": prec,
                "set": rng.randint(2, 99)}
    if kind == "fidelity":
        return {"kind": kind, "circuit": "w42", "precision": prec, "n": _log(rng, 10000, 2097169),
                "p": _noise(rng, 5e-4, 2e-3)}
    if kind == "grad":
        return {"kind": kind, "precision": "fp64", "n": _log(rng, 1000, 100003)}
    q = rng.randint(3, 7)
    return {"kind": kind, "circuit_seed": rng.randint(700, 799), "qubits": q, "ops": 50 + 6 * q + rng.randint(0, 30),
            "params": rng.randint(3, 9), "p": _noise(rng, 5e-3, 3e-2), "precision": prec,
            "n": _log(rng, 256, 8000 if q <= 5 else 2000)}


def _noise(rng, lo, hi):
    return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))


# ------------------------------------------------------------------ circuits
@functools.lru_cache(maxsize=64)
def _named(name, circuit_seed=0, qubits=0, blocks=0, w=0):
    if name == "random40":
        c = C.random_circuit(4040, 40, 400, t_frac=0.08, meas_frac=0.2, detectors=True, mpp_frac=0.05)
        c.cap = 256
    elif name == "window":
        c, _ = C.windowed(circuit_seed, n_data=qubits - 4, n_anc=4, blocks=blocks, w=w,
                          n_cliff=max(20, 2 * (qubits - 4)), checks=4)
    else:
        c, _ = C.workload(name)
    return c, c.array()


def _circuit(case):
    if case["kind"] == "grad":
        return _named("w42rz")
    return _named(case["circuit"], *(case.get(k, 0) for k in ("circuit_seed", "qubits", "blocks", "w")))


@functools.lru_cache(maxsize=8)
def _batch(which, circuits, mean):
    return [(c, c.array(), noise, n) for c, noise, n in C.batch_of_windowed(which, circuits, mean)]


@functools.lru_cache(maxsize=16)
def _param_circuit(seed, qubits, ops, params):
    c, _ = C.random_param_circuit(seed, qubits, ops, params)
    return c, c.array()


def _first(seed):
    return (int(seed) * 2654435761) % (1 << 40)


def prepare(case, seed):
    dev = torch.device("cuda")
    st = {"case": case, "seed": int(seed), "first": _first(seed), "kind": case["kind"]}
    if case["kind"] == "batch":
        items = _batch(case["set"], case["circuits"], case["mean"])
        st["circs"] = [S.soft_compile_circuit(a, c.n, noise, c.cap) for c, a, noise, _ in items]
        st["n"] = [n for _, _, _, n in items]
        st["firsts"] = [st["first"]] * len(items)
        return st
    if case["kind"] == "train":
        c, a = _param_circuit(case["circuit_seed"], case["qubits"], case["ops"], case["params"])
        st["circ"] = S.soft_compile_circuit(a, c.n, C.Noise.uniform(case["p"]), c.cap)
        st["theta"] = _theta(case, seed).to(dev).requires_grad_(True)
        return st
    c, a = _circuit(case)
    if case["kind"] == "sweep":  # the op list in host memory; the call compiles it
        st.update(ops=a, qubits=c.n, cap=c.cap, noise=C.Noise.uniform(case["p"]))
        return st
    st["circ"] = S.soft_compile_circuit(a, c.n, C.Noise.uniform(case.get("p", 1e-3)), c.cap)
    if case["kind"] == "grad":  # the angles as an optimiser hands them over: around pi/4
        st["theta"] = C.rz_thetas(int(seed), 72)
    elif case.get("records"):
        st["status"] = torch.empty(case["n"], dtype=torch.uint8, device=dev)
        st["rec"] = torch.empty((case["n"], st["circ"].info["record_words"]), dtype=torch.int64, device=dev)
    return st


def _theta(case, seed):
    g = torch.Generator().manual_seed(int(seed))
    t = torch.rand(case["params"], generator=g, dtype=torch.float64) * (2 * math.pi) - math.pi
    return t.to(torch.float32 if case["precision"] == "fp32" else torch.float64)


def _tally(t, names=TALLY):
    return {k: t[k] for k in names}


def run(st):
    case, kind, prec = st["case"], st["kind"], st["case"]["precision"]
    if kind == "shots":
        kw = {}
        if case["records"]:
            kw = dict(record_mode=S.REC_ALL, d_records=st["rec"].data_ptr(), d_status=st["status"].data_ptr())
        r = S.soft_run_shots(st["circ"], case["n"], st["first"], st["seed"], precision=prec, **kw)
        out = _tally(S.soft_tally(r))
        r.free()
        if case["records"]:
            out.update(status=st["status"], records=st["rec"])
        return out
    if kind == "sweep":
        c = S.soft_compile_circuit(st["ops"], st["qubits"], st["noise"], st["cap"])
        r = S.soft_run_shots(c, case["n"], st["first"], st["seed"], precision=prec)
        out = _tally(S.soft_tally(r))
        r.free()
        c.free()
        return out
    if kind == "batch":
        r = S.soft_run_batch(st["circs"], st["n"], st["firsts"], st["seed"], precision=prec)
        t = [S.soft_tally_batch(r, i) for i in range(len(st["n"]))]
        r.free()
        return {"tallies": np.array([[x[k] for k in TALLY] for x in t], dtype=np.int64)}
    if kind == "fidelity":
        r = S.soft_run_shots(st["circ"], case["n"], st["first"], st["seed"], precision=prec, fidelity=True)
        out = _tally(S.soft_tally(r), TALLY + ("sum_fidelity", "sum_weight"))
        r.free()
        return out
    if kind == "grad":
        fid, pacc, grad, status, sums = S.soft_fidelity_grad(st["circ"], st["theta"], case["n"], st["first"],
                                                             st["seed"], prec, sums=True)
        return {"fid": fid, "pacc": pacc, "grad": grad, "status": status, "sums": sums}
    # one step: the post-selected infidelity over the patterns (acceptances as weights), its gradient
    th = st["theta"]
    th.grad = None
    fid, pacc, status = PostSelectedFidelity.apply(th, st["circ"], case["n"], st["first"], st["seed"], prec)
    loss = 1.0 - (pacc * fid).sum() / pacc.sum()
    loss.backward()
    return {"loss": loss.detach(), "fid": fid.detach(), "pacc": pacc, "status": status, "grad": th.grad}


# ------------------------------------------------------------------ work
def _program_bytes(a):
    sites = int(np.isin(a["op"], C.ONE_Q + C.TWO_Q + (C.M, C.R, C.MR)).sum())
    events = int((a["op"] > C.CZ).sum())
    return 64.0 * events + 176.0 * sites, sites


def _shot_flops(case, a, sites):
    """Floating-point operations a shot cannot do without: 14 per entry that a rotation writes (two
    complex products and a sum), 4 per entry that a measurement reads. Until its first error a shot
    equals the noiseless run, which is computed once; a post-selected shot then lives about a block
    of the circuit, until a check catches its error. Without post-selection it runs to the end."""
    rot, meas = int(np.isin(a["op"], (C.T, C.T_DAG, C.RZ)).sum()), int(np.isin(a["op"], (C.M, C.R, C.MR)).sum())
    if case.get("circuit") in ("tiny6", "random40"):
        return (1.0 - (1.0 - case["p"]) ** sites) * (14.0 * 4 * rot + 4.0 * 4 * meas)
    w, checks = {"w42": (4, 4), "w97": (6, 8)}.get(case.get("circuit"), (case.get("w", 4), 4))
    block = 14.0 * 2 * (2 ** (w + 1) - 2) + 4.0 * 2 * checks * 2 ** w
    return (1.0 - (1.0 - case.get("p", 1e-3)) ** sites) * block


def work(case):
    if case["kind"] == "batch":
        b = f = 0.0
        for c, a, noise, n in _batch(case["set"], case["circuits"], case["mean"]):
            pb, sites = _program_bytes(a)
            w = int(round(math.log(c.cap, 4)))
            b += pb + 40.0
            f += n * _shot_flops({"kind": "shots", "p": noise.p1, "w": w}, a, sites)
        return {"bytes": b, "flops": f}
    if case["kind"] == "train":
        c, a = _param_circuit(case["circuit_seed"], case["qubits"], case["ops"], case["params"])
        # forward, one adjoint sweep and the derivative of each angle, on the final map size
        rot = int((a["op"] == C.RZ).sum())
        f = case["n"] * 3.0 * 14.0 * rot * 2 ** case["qubits"]
        return {"bytes": _program_bytes(a)[0] + case["n"] * (17.0 + 8.0 * case["params"]), "flops": f}
    c, a = _circuit(case)
    pb, sites = _program_bytes(a)
    if case["kind"] == "grad":
        # 94 % of the patterns are rejected within about a block; the rest go forward and back once
        whole = 18 * (14.0 * 60 + 4.0 * 128)
        return {"bytes": pb + case["n"] * (17.0 + 8.0 * 72), "flops": case["n"] * (whole / 18 + 0.06 * 3.0 * whole)}
    out = case["n"] * (1.0 + 8.0 * -(-_records(a) // 64)) if case.get("records") else 40.0
    return {"bytes": pb + out, "flops": case["n"] * _shot_flops(case, a, sites)}


def _records(a):
    mpp_end = (a["op"] == C.MPP) & ((a["flags"] & C.MPP_MORE) == 0)
    return int(np.isin(a["op"], (C.M, C.MR)).sum() + mpp_end.sum())


# ------------------------------------------------------------------ the same in 64 bits, dense
_P = [np.eye(2, dtype=complex), np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]], complex),
      np.array([[1, 0], [0, -1]], complex)]


def _philox(seed, shots, idx):
    """Philox4x32-10 (Salmon et al. 2011), counter (shot, shot >> 32, 0, idx), key = seed, over arrays."""
    m = np.uint64(0xFFFFFFFF)
    sh = np.uint64(32)
    c = [shots & m, shots >> sh, np.zeros_like(shots), idx.astype(np.uint64)]
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(b >> sh) ^ c[1] ^ k0, b & m, (a >> sh) ^ c[3] ^ k1, a & m]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m, (k1 + np.uint64(0xBB67AE85)) & m
    return c


def _patterns(case, ops, seed):
    """The Pauli code (0: none) of every noise site of every pattern: geometric gaps of one rate."""
    n, p = case["n"], case["p"]
    sites, quiet = [], False
    for i, o in enumerate(ops):
        if o[0] in (C.NOISELESS_BEGIN, C.NOISELESS_END):
            quiet = o[0] == C.NOISELESS_BEGIN
        elif not quiet and o[0] == C.M:
            sites.append((i, "flip"))
        elif not quiet and o[0] in C.ONE_Q + C.TWO_Q:
            sites.append((i, "two" if o[0] in C.TWO_Q else "one"))
    shots = np.arange(n, dtype=np.uint64) + np.uint64(_first(seed))
    codes = np.zeros((len(sites), n), dtype=np.int64)
    ladder = -np.expm1(np.arange(1, len(sites) + 1) * math.log1p(-p))  # P(gap <= g)
    at, k, live = np.zeros(n, dtype=np.int64), np.zeros(n, dtype=np.int64), np.arange(n)
    while live.size:
        w = _philox(int(seed), shots[live], k[live])
        k[live] += 1
        u = (w[0].astype(np.float64) + w[1].astype(np.float64) * 2.0 ** 32) * 2.0 ** -64
        s = at[live] + np.searchsorted(ladder, u, side="right")
        hit = s < len(sites)
        live, s, w2 = live[hit], s[hit], w[2][hit]
        at[live] = s + 1
        kinds = np.array([{"flip": 0, "one": 3, "two": 15}[t] for _, t in sites])[s].astype(np.uint64)
        codes[s, live] = np.where(kinds == 0, 1, (w2 * kinds >> np.uint64(32)).astype(np.int64) + 1)
    return {i: (t, codes[j]) for j, (i, t) in enumerate(sites)}


def _on(psi, n, q, u):
    """One-qubit matrix u (2 x 2, or one per pattern) on qubit q of psi (patterns x 2^n)."""
    t = psi.reshape(len(psi), 2 ** (n - 1 - q), 2, 2 ** q)
    return np.einsum("pab,pibj->piaj" if u.ndim == 3 else "ab,pibj->piaj", u, t).reshape(psi.shape)


def _linear(psi, n, o, angle, noise, dag=False):
    """One op (and its noise) of the post-selected circuit, or its adjoint, without renormalising."""
    idx = np.arange(2 ** n)
    table = np.array(_P)

    def error(v):
        if noise is None:
            return v
        kind, code = noise
        if kind == "two":
            return _on(_on(v, n, o[2], table[code >> 2]), n, o[3], table[code & 3])
        return _on(v, n, o[2], table[code])

    def body(v):
        op, q0, q1 = o[0], o[2], o[3]
        if op == C.CX:
            return v[:, idx ^ (((idx >> q0) & 1) << q1)]
        if op == C.CZ:
            return v * np.where((idx >> q0) & (idx >> q1) & 1, -1.0, 1.0)
        if op == C.M:
            return v * ((idx >> q0) & 1 == angle)
        u = {C.H: (_P[1] + _P[3]) / math.sqrt(2), C.S: np.diag([1, 1j]), C.S_DAG: np.diag([1, -1j]), C.X: _P[1],
             C.Y: _P[2], C.Z: _P[3], C.RZ: np.diag(np.exp([-0.5j * angle, 0.5j * angle]))}[op]
        return _on(v, n, q0, u.conj().T if dag else u)

    first = o[0] == C.M  # a flip comes before its measurement, a gate's error after it
    if dag:
        first = not first
    return body(error(psi)) if first else error(body(psi))


def exact(case, seed):
    if case["kind"] != "train" or case["n"] * 2 ** case["qubits"] > 1 << 19:
        return None
    c, _ = _param_circuit(case["circuit_seed"], case["qubits"], case["ops"], case["params"])
    n, theta = c.n, _theta(case, seed).double().numpy()
    want, seen = {}, []  # the outcome each record is projected onto; observed records come last
    for o in c.ops:
        if o[0] == C.DETECTOR:
            want[o[6][0]] = 1 if o[1] & C.FLAG_INVERT else 0
        elif o[0] == C.OBSERVABLE:
            seen.append(o[6][0])
    noise = _patterns(case, c.ops, seed)
    steps, record = [], 0
    for i, o in enumerate(c.ops):
        if o[0] == C.M:
            steps.append((o, want.get(record, 0), noise.get(i), record in seen))
            record += 1
        elif o[0] in C.ONE_Q + C.TWO_Q:
            ang = (-1.0 if o[1] & 1 else 1.0) * theta[o[4] - 1] if o[0] == C.RZ else 0.0
            steps.append((o, ang, noise.get(i), False))
    psi = np.zeros((case["n"], 2 ** n), complex)
    psi[:, 0] = 1.0
    after, cut = [], None
    for k, (o, ang, err, obs) in enumerate(steps):
        if obs and cut is None:
            cut = k
            pre = psi
        psi = _linear(psi, n, o, ang, err)
        after.append(psi)
    norm = lambda v: (np.abs(v) ** 2).sum(1)  # noqa: E731
    acc = norm(pre)
    acc = np.where(acc > 1e-20, acc, 0.0)
    safe = np.where(acc > 0, acc, 1.0)
    fid = norm(psi) / safe * (acc > 0)
    grad = np.zeros((case["n"], case["params"]))
    lam = psi
    for k in range(len(steps) - 1, -1, -1):
        o, ang, err, _ = steps[k]
        if k + 1 == cut:
            lam = lam - fid[:, None] * pre
        if o[0] == C.RZ:
            # d/dtheta of exp(-i s theta Z / 2), with the error that follows it carried along
            sgn = -1.0 if o[1] & 1 else 1.0
            z = np.where((np.arange(2 ** n) >> o[2]) & 1, -1.0, 1.0)
            before = after[k - 1] if k else np.eye(1, 2 ** n, dtype=complex).repeat(case["n"], 0)
            lam = _linear(lam, n, o, ang, err, dag=True)
            grad[:, o[4] - 1] += sgn * np.imag((lam.conj() * z * before).sum(1)) / safe * (acc > 0)
        else:
            lam = _linear(lam, n, o, ang, err, dag=True)
    loss = 1.0 - (acc * fid).sum() / acc.sum()
    weights = acc / acc.sum()
    return {"loss": np.float64(loss), "fid": fid, "pacc": acc, "status": None, "grad": -(weights[:, None] * grad).sum(0)}
