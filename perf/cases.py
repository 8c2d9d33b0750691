"""Timed cases: what a user of the simulator has it do, through the package's public entry points.

A state is psi = C|MPS>.  The cases cover whole circuits (one call per gate list, single and batched, FP64
and precision form), the same work gate by gate, pure Clifford circuits, the class scoring on a caller's
tensor (with and without a handle), the readouts and the phase gradient.  Circuits of the benchmark family
(brickwork of random two-qudit Cliffords with T gates spread over the layers) use
``sp4_images``; circuits whose outputs are also computed densely (``exact``) use the named gates.
"""
import functools
import itertools
import math
import random

import numpy as np
import torch

import paper_2511_06672_gb300 as gc


def listed():
    return [
        # one class search on a small qubit bond, device buffers: the smallest call of the library
        {"name": "score_qubit_small", "kind": "score", "via": "noalloc", "d": 2, "chi_l": 2, "chi_r": 3,
         "score_kind": 0},
        # the same entry on a big, ragged qutrit bond (its limit is chi 27)
        {"name": "score_qutrit_large", "kind": "score", "via": "noalloc", "d": 3, "chi_l": 27, "chi_r": 25,
         "score_kind": 0},
        # the handle's class scores on a host tensor, bond-dimension criterion
        {"name": "score_handle_ragged", "kind": "score", "via": "handle", "d": 3, "chi_l": 9, "chi_r": 14,
         "score_kind": 2},
        # stabilizer circuit: a wide brickwork with no T gate, only the tableau moves
        {"name": "clifford_wide", "kind": "clifford", "d": 3, "n": 96, "layers": 24},
        # interactive use: one call per gate on a small register
        {"name": "gate_by_gate", "kind": "gates", "d": 2, "n": 10, "layers": 8, "t": 5},
        # the benchmark's qubit circuits: 32 qubits, one launch
        {"name": "run_qubit", "kind": "run", "d": 2, "n": 32, "layers": 24, "t": 32, "chi_max": 256, "batch": 1,
         "cluster": 4, "precision": 0},
        # the benchmark's qutrit circuits: 32 qutrits, one launch
        {"name": "run_qutrit", "kind": "run", "d": 3, "n": 32, "layers": 24, "t": 26, "chi_max": 256, "batch": 1,
         "cluster": 16, "precision": 0},
        # many independent uneven circuits in one launch
        {"name": "run_batch", "kind": "run", "d": 3, "n": 20, "layers": 16, "t": 15, "chi_max": 128, "batch": 48,
         "cluster": 4, "precision": 0},
        # the precision form (FP32 contractions) on a mid-sized qutrit circuit
        {"name": "run_precision", "kind": "run", "d": 3, "n": 24, "layers": 24, "t": 20, "chi_max": 128, "batch": 1,
         "cluster": 16, "precision": 1},
        # a training step: forward run and adjoint gradient of a parametrised qubit circuit (its observable, a Pauli
        # string, is Hermitian)
        {"name": "gradient", "kind": "gradient", "d": 2, "n": 12, "layers": 10, "t": 8, "chi_max": 64},
        # observables of a finished run: strings' expectation values and the Schmidt values of a bond
        {"name": "observables", "kind": "observables", "d": 3, "n": 32, "layers": 24, "t": 20, "chi_max": 256,
         "strings": 16},
        # dense state of a small register
        {"name": "statevector", "kind": "statevector", "d": 3, "n": 8, "layers": 8, "t": 3, "disentangle": False},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["score", "score", "clifford", "gates", "run", "run", "run", "gradient", "observables",
                       "statevector"])
    d = rng.choice([2, 3])
    if kind == "score":
        via = rng.choice(["noalloc", "handle"])
        top = 27 if d == 3 else 40
        return {"kind": kind, "via": via, "d": d, "chi_l": _logint(rng, 1, top), "chi_r": _logint(rng, 2, top),
                "score_kind": 0 if via == "noalloc" else rng.choice([0, 1, 2])}
    if kind == "clifford":
        return {"kind": kind, "d": d, "n": _logint(rng, 6, 128), "layers": rng.randint(4, 24)}
    if kind == "gates":
        return {"kind": kind, "d": d, "n": rng.randint(4, 12 if d == 2 else 7), "layers": rng.randint(4, 8),
                "t": rng.randint(1, 4)}
    if kind == "run":
        batch = rng.choice([1, 1, _logint(rng, 2, 48)])
        n = _logint(rng, 8, 32) if batch == 1 else _logint(rng, 8, 20)
        t = rng.randint(max(1, n // 3), 3 * n // 4) if d == 3 else rng.randint(n // 3, n)
        return {"kind": kind, "d": d, "n": n, "layers": rng.randint(8, 24), "t": t,
                "chi_max": 256 if batch == 1 else 128, "batch": batch,
                "cluster": rng.choice([8, 16]) if batch == 1 else rng.choice([2, 4, 8]),
                "precision": rng.choice([0, 0, 1])}
    if kind == "gradient":
        n = rng.randint(5, 12)
        return {"kind": kind, "d": 2, "n": n, "layers": rng.randint(6, 10), "t": rng.randint(3, 8),
                "chi_max": 2 ** (n // 2)}
    if kind == "observables":
        n = _logint(rng, 10, 32)
        return {"kind": kind, "d": d, "n": n, "layers": rng.randint(12, 24), "t": rng.randint(n // 3, 2 * n // 3),
                "chi_max": 256, "strings": rng.randint(4, 24)}
    return {"kind": kind, "d": d, "n": rng.randint(5, 12 if d == 2 else 8), "layers": rng.randint(4, 8),
            "t": rng.randint(1, 4), "disentangle": rng.random() < 0.4}


# ------------------------------------------------------------------------------------------ circuits
ONE_QUDIT = {"H": gc.GATE_H, "S": gc.GATE_S, "X": gc.GATE_X, "Z": gc.GATE_Z}
SP4_ORDER = {2: 720, 3: 51840}


def t_phases(d):
    return (0.0, math.pi / 4) if d == 2 else (0.0, 2 * math.pi / 9, -2 * math.pi / 9)


def _after_layer(layers, t):
    """Layer after which each of t T gates comes: spread evenly, the last one after the last layer."""
    return [((k + 1) * layers + t - 1) // t - 1 for k in range(t)]


def brickwork(d, n, layers, t, rng):
    """("C2", q, sp_index, shift) and ("T", site, phases) gates of the benchmark family."""
    gates, after = [], _after_layer(layers, t) if t else []
    for layer in range(layers):
        for q in range(layer % 2, n - 1, 2):
            gates.append(("C2", q, rng.randrange(SP4_ORDER[d]), tuple(rng.randrange(d) for _ in range(4))))
        gates += [("T", rng.randrange(n), t_phases(d)) for a in after if a == layer]
    return gates


def named_circuit(d, n, layers, t, rng, parametrised=False):
    """The same family written in named gates: on every pair a scrambler of H, S, X, Z and both SUMs."""
    gates, after = [], _after_layer(layers, t)
    for layer in range(layers):
        for q in range(layer % 2, n - 1, 2):
            for control, target in rng.sample([(q, q + 1), (q + 1, q)], 2):
                for site in (q, q + 1):
                    gates += [(g, site) for g in rng.choice((("H",), ("S", "H"), ("H", "S"), ("X", "H"), ("Z", "S")))]
                gates.append(("SUM", control, target))
        for _ in (a for a in after if a == layer):
            th = rng.uniform(0.3, 2.8)
            phases = t_phases(d) if not parametrised else ((0.0, th) if d == 2 else (0.0, th, -th))
            gates.append(("T", rng.randrange(n), phases))
    return gates


@functools.lru_cache(maxsize=1 << 16)
def _images(d, gate):
    if gate[0] == "C2":
        return gc.sp4_images(d, gate[2], gate[3])
    return gc.named_images(d, gc.GATE_SUM if gate[0] == "SUM" else ONE_QUDIT[gate[0]])


def to_ops(d, gates, disentangle=True):
    rows = []
    for g in gates:
        op = np.zeros((), dtype=gc.OP_DTYPE)
        if g[0] == "T":
            op["kind"], op["q0"], op["q1"] = gc.OP_NONCLIFFORD, g[1], -1
            op["phases"][: len(g[2])] = g[2]
        else:
            img = _images(d, ("C2", 0) + g[2:] if g[0] == "C2" else (g[0],))
            op["kind"], op["q0"] = gc.OP_CLIFFORD, g[1]
            op["q1"] = g[1] + 1 if g[0] == "C2" else (g[2] if g[0] == "SUM" else -1)
            op["img"][: len(img)] = img
        rows.append(op)
        if g[0] == "T" and disentangle:
            op = np.zeros((), dtype=gc.OP_DTYPE)
            op["kind"] = gc.OP_DISENTANGLE
            rows.append(op)
    return np.array(rows, dtype=gc.OP_DTYPE)


def evolved_strings(d, n, gates):
    """For every qudit q the exponents (x, z) of the string Z_q becomes under the Cliffords of the circuit, and
    the number of its T gates that do not commute with it on the way.  <psi|W|psi> of such a string is rarely 0."""
    w = np.zeros((n, 2 * n), dtype=np.int64)
    w[np.arange(n), n + np.arange(n)] = 1
    met = np.zeros(n, dtype=np.int64)
    for g in gates:
        if g[0] == "T":
            met += w[:, g[1]] != 0
            continue
        img = _images(d, ("C2", 0) + g[2:] if g[0] == "C2" else (g[0],))
        if len(img) == 20:
            q0, q1 = g[1], g[1] + 1 if g[0] == "C2" else g[2]
            cols, m = [q0, n + q0, q1, n + q1], np.asarray(img).reshape(4, 5)[:, :4]
        else:
            cols, m = [g[1], n + g[1]], np.asarray(img).reshape(2, 3)[:, :2]
        w[:, cols] = w[:, cols] @ m % d
    return w[:, :n].astype(np.int32), w[:, n:].astype(np.int32), met


# ------------------------------------------------------------------------------- two-site tensors
@functools.lru_cache(maxsize=None)
def class_matrices(d):
    """The two-qudit Cliffords modulo single-qudit Cliffords after them, as 4x4 symplectic matrices: a class is
    the plane its first two rows span (the other two span the complement); smallest member, identity first."""
    vecs = [np.array(v) for v in itertools.product(range(d), repeat=4)]
    code = {tuple(v): i for i, v in enumerate(vecs)}
    form = lambda u, v: int(u[0] * v[1] - u[1] * v[0] + u[2] * v[3] - u[3] * v[2]) % d  # noqa: E731
    lam = np.array([[form(u, v) for v in vecs] for u in vecs])

    def smallest_pair(members):
        a = members[1]
        return a, next(b for b in members if lam[a][b] == 1)

    found = {}
    for a in range(1, len(vecs)):
        for b in range(1, len(vecs)):
            if lam[a][b] != 1:
                continue
            plane = frozenset(code[tuple((i * vecs[a] + j * vecs[b]) % d)] for i in range(d) for j in range(d))
            if plane not in found:
                rest = [v for v in range(len(vecs)) if all(lam[u][v] == 0 for u in plane)]
                found[plane] = smallest_pair(sorted(plane)) + smallest_pair(rest)
    local = frozenset(code[(i, j, 0, 0)] for i in range(d) for j in range(d))
    rows = [s for plane, s in found.items() if plane != local]
    return [np.eye(4, dtype=np.int64)] + [np.stack([vecs[i] for i in s]) for s in sorted(rows)]


def weyl_matrix(d, v, nq=2):
    """X^v0 Z^v1 (x) X^v2 Z^v3, with the phase that makes its order d."""
    w = np.exp(2j * np.pi / d)
    out = np.ones((1, 1), dtype=np.complex128)
    for q in range(nq):
        x, z = int(v[2 * q]), int(v[2 * q + 1])
        m = np.roll(np.eye(d), x, axis=0) @ np.diag(w ** (z * np.arange(d)))
        out = np.kron(out, m * (1j ** (x * z) if d == 2 else 1.0))
    return out


@functools.lru_cache(maxsize=None)
def class_unitaries(d):
    out = []
    for s in class_matrices(d):
        x0, z0, x1, z1 = (weyl_matrix(d, s[:, k]) for k in range(4))
        power = np.linalg.matrix_power
        proj = sum(power(z0, a) @ power(z1, b) for a in range(d) for b in range(d)) / d ** 2
        v = proj[:, int(np.argmax(np.linalg.norm(proj, axis=0)))]
        v = v / np.linalg.norm(v)
        out.append(np.stack([power(x0, a) @ power(x1, b) @ v for a in range(d) for b in range(d)], axis=1))
    return np.array(out)


def bond_tensor(d, chi_l, chi_r, seed):
    """A two-site tensor (chi_l, d, d, chi_r) as a sweep meets it: a decaying Schmidt spectrum of limited rank, then
    a random two-qudit Clifford that the search can undo."""
    rng = np.random.default_rng(seed)
    rank = max(1, min(chi_l * d, chi_r * d) // d)
    g = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
    a = np.linalg.qr(g(chi_l * d, rank))[0]
    b = np.linalg.qr(g(d * chi_r, rank))[0].T
    lam = np.exp(-0.15 * np.arange(rank) * rng.uniform(0.5, 1.5))
    th = (a * lam / np.linalg.norm(lam)) @ b
    u = class_unitaries(d)
    u = u[rng.integers(len(u))]
    th = np.einsum("uv,avb->aub", u, th.reshape(chi_l, d * d, chi_r))
    return np.ascontiguousarray(th.reshape(chi_l, d, d, chi_r))


# ------------------------------------------------------------------------------------------ prepare
class _State:
    def __init__(self, **kw):
        self.__dict__.update(kw)


def _batch_sizes(case):
    """Qudit counts of a batch: from two thirds of the largest up to it."""
    n, b = case["n"], case["batch"]
    return [n] if b == 1 else [n - (i * (n // 3 + 1)) // b for i in range(b)]


def prepare(case, seed):
    rng = random.Random(seed)
    d, kind = case["d"], case["kind"]
    if kind == "score":
        th = bond_tensor(d, case["chi_l"], case["chi_r"], seed)
        if case["via"] == "handle":
            chi = max(case["chi_l"], case["chi_r"])
            n = 2 * max(1, math.ceil(math.log(chi) / math.log(d) - 1e-9)) + 2
            return _State(kind="score_handle", theta=th,
                          sim=gc.Simulator(n, d, chi_max=chi, score_kind=case["score_kind"]))
        k = gc.num_candidates(d)
        dev = lambda dtype, m: torch.empty(m, dtype=dtype, device="cuda")  # noqa: E731
        return _State(kind="score_noalloc", case=case, theta=torch.from_numpy(th).cuda(), s2=dev(torch.float64, k),
                      vn=dev(torch.float64, k), choice=dev(torch.int32, 3))
    if kind == "clifford":
        gates = brickwork(d, case["n"], case["layers"], 0, rng)
        return _State(kind=kind, sim=gc.Simulator(case["n"], d, chi_max=8), ops=to_ops(d, gates))
    if kind == "gates":
        n = case["n"]
        gates = named_circuit(d, n, case["layers"], case["t"], rng)
        return _State(kind=kind, sim=gc.Simulator(n, d, chi_max=d ** (n // 2)), gates=gates,
                      strings=evolved_strings(d, n, gates))
    if kind == "run":
        sizes = _batch_sizes(case)
        ops, begin, strings = [], [0], []
        for n in sizes:
            gates = brickwork(d, n, case["layers"], min(case["t"], case["t"] * n // case["n"] + 1), rng)
            ops.append(to_ops(d, gates))
            begin.append(begin[-1] + len(ops[-1]))
            strings.append(evolved_strings(d, n, gates))
        sim = gc.Simulator(sizes if case["batch"] > 1 else sizes[0], d, chi_max=case["chi_max"],
                           cluster_size=case["cluster"], precision=case["precision"])
        return _State(kind=kind, sim=sim, ops=np.concatenate(ops), begin=begin if case["batch"] > 1 else None,
                      strings=strings)
    if kind == "gradient":
        n = case["n"]
        gates, x, z = parametrised(case, rng)
        sim = gc.Simulator(n, d, chi_max=case["chi_max"], snapshot_entries=1 << 20, snapshot_max_gates=case["t"])
        return _State(kind=kind, sim=sim, ops=to_ops(d, gates), x=x, z=z)
    if kind == "observables":
        n = case["n"]
        gates = brickwork(d, n, case["layers"], case["t"], rng)
        sim = gc.Simulator(n, d, chi_max=case["chi_max"], cluster_size=16)
        sim.run(to_ops(d, gates))
        sim.sync()
        x, z, _ = evolved_strings(d, n, gates)
        # sums of neighbouring strings too: products of the observables above
        x = np.concatenate([x, (x + np.roll(x, 1, 0)) % d])[: case["strings"]]
        z = np.concatenate([z, (z + np.roll(z, 1, 0)) % d])[: case["strings"]]
        return _State(kind=kind, sim=sim, x=x, z=z, bond=n // 2)
    n = case["n"]
    gates = named_circuit(d, n, case["layers"], case["t"], rng)
    sim = gc.Simulator(n, d, chi_max=d ** (n // 2))
    sim.run(to_ops(d, gates, case["disentangle"]))
    sim.sync()
    return _State(kind=kind, sim=sim)


# ---------------------------------------------------------------------------------------------- run
def run(s):
    sim = getattr(s, "sim", None)
    if s.kind == "score_noalloc":
        c = s.case
        gc.score_theta_noalloc(c["d"], c["chi_l"], c["chi_r"], s.theta, s.s2, s.vn, s.choice,
                               stream=torch.cuda.current_stream())
        return {"s2": s.s2, "vn": s.vn, "choice": s.choice}
    if s.kind == "score_handle":
        s2, vn, choice, evaluated = sim.score_theta(s.theta)
        return {"s2": s2, "vn": vn, "choice": choice, "evaluated": evaluated}
    if s.kind == "clifford":
        sim.reset()
        sim.run(s.ops)
        (e, p), (ie, ip) = sim.tableau(), sim.inverse_tableau()
        return {"exps": e, "phase": p, "inv_exps": ie, "inv_phase": ip}
    if s.kind == "gates":
        sim.reset()
        for g in s.gates:
            if g[0] == "T":
                sim.apply_nonclifford(g[1], g[2])
                sim.disentangle()
            elif g[0] == "SUM":
                sim.apply_named(gc.GATE_SUM, g[1], g[2])
            else:
                sim.apply_named(ONE_QUDIT[g[0]], g[1])
        x, z, _ = s.strings
        return {"expect": np.array([sim.expect_weyl(x[q], z[q]) for q in range(len(x))]),
                "bond_dims": np.array(sim.bond_dims())}
    if s.kind == "run":
        sim.reset()
        sim.run(s.ops, s.begin)
        tableaux = [sim.tableau(c) for c in range(sim.batch)]
        dims = [sim.bond_dims(c) for c in range(sim.batch)]
        picked = range(0, sim.batch, max(1, sim.batch // 8))
        expect = [sim.expect_weyl(s.strings[c][0][q], s.strings[c][1][q], c)
                  for c in picked for q in range(8 if sim.batch == 1 else 2)]
        return {"bond_dims": np.concatenate([np.array(v) for v in dims]),
                "exps": np.concatenate([e.reshape(-1) for e, _ in tableaux]),
                "phase": np.concatenate([p for _, p in tableaux]), "expect": np.array(expect)}
    if s.kind == "gradient":
        sim.reset()
        sim.run(s.ops)
        value, grad = sim.expect_gradient(s.x, s.z)
        return {"value": value, "grad": grad}
    if s.kind == "observables":
        return {"expect": np.array([sim.expect_weyl(x, z) for x, z in zip(s.x, s.z)]),
                "schmidt": sim.schmidt_values(s.bond)}
    return {"psi": sim.statevector()}


# --------------------------------------------------------------------------------------------- work
def _class_flops(d, chi_l, chi_r):
    """FP64 flops of one exact class score: Q theta, its Gram, the reduction of the Gram."""
    r, c = chi_l * d, chi_r * d
    m, big = min(r, c), max(r, c)
    return 8.0 * d * d * r * c + 4.0 * m * (m + 1) * big + 16.0 / 3.0 * m ** 3


def _circuit_work(d, n, layers, t):
    """A circuit at its lowest bond dimensions: the gate list in, the tableau out; per T gate one sweep that scores
    every class on bonds of dimension d."""
    gates = layers * (n - 1) // 2 + 2 * t
    classes = d * d * (d * d + 1)
    return {"bytes": 128.0 * gates + 2 * (4 * n * n + 2 * n),
            "flops": t * (n - 1) * classes * _class_flops(d, d, d) + layers * (n // 2) * 20.0 * n}


def work(case):
    d, kind = case["d"], case["kind"]
    if kind == "score":
        k, cl, cr = d * d * (d * d + 1), case["chi_l"], case["chi_r"]
        return {"bytes": 16.0 * cl * d * d * cr + 16.0 * k, "flops": k * _class_flops(d, cl, cr)}
    n, layers = case["n"], case["layers"]
    if kind == "clifford":
        return _circuit_work(d, n, layers, 0)
    if kind == "run":
        parts = [_circuit_work(d, m, layers, min(case["t"], case["t"] * m // n + 1)) for m in _batch_sizes(case)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    if kind == "gates":
        return _circuit_work(d, n, layers, case["t"])
    if kind == "gradient":
        w = _circuit_work(d, n, layers, case["t"])
        return {"bytes": w["bytes"], "flops": 2 * w["flops"]}
    if kind == "observables":   # transfer matrices at bond dimension d
        return {"bytes": 16.0 * n * d ** 3 + 2.0 * n * case["strings"],
                "flops": 16.0 * case["strings"] * n * d ** 4}
    # C as one two-qudit gate per pair of qudits on the dense vector
    return {"bytes": 16.0 * d ** n, "flops": 8.0 * d ** n * d * d * n * (n - 1) / 2}


# -------------------------------------------------------------------------------------------- exact
def _one_site(psi, m, q):
    return np.moveaxis(np.tensordot(m, psi, axes=(1, q)), 0, q)


def _gate_matrix(d, name):
    j = np.arange(d)
    w = np.exp(2j * np.pi / d)
    if name == "H":
        return w ** np.outer(j, j) / math.sqrt(d)
    if name == "S":
        return np.diag([1, 1j]) if d == 2 else np.diag(w ** (j * (j - 1) // 2))
    return np.roll(np.eye(d), 1, axis=0) if name == "X" else np.diag(w ** j)


def _sum_gate(d, psi, control, target):
    out = np.empty_like(psi)
    for i in range(d):
        at = [slice(None)] * psi.ndim
        at[control] = i
        out[tuple(at)] = np.roll(psi[tuple(at)], i, axis=target - (target > control))
    return out


def dense(d, n, gates, t_gates=True):
    """The state after the circuit, and the states right after each T gate."""
    psi = np.zeros((d,) * n, dtype=np.complex128)
    psi[(0,) * n] = 1.0
    snaps = []
    for g in gates:
        if g[0] == "T":
            if t_gates:
                psi = _one_site(psi, np.diag(np.exp(1j * np.array(g[2]))), g[1])
                snaps.append(psi)
        elif g[0] == "SUM":
            psi = _sum_gate(d, psi, g[1], g[2])
        else:
            psi = _one_site(psi, _gate_matrix(d, g[0]), g[1])
    return psi, snaps


def dense_weyl(d, psi, x, z):
    w = np.exp(2j * np.pi / d)
    for q in range(psi.ndim):
        if z[q]:
            psi = _one_site(psi, np.diag(w ** (z[q] * np.arange(d))), q)
        if x[q]:
            psi = np.roll(psi, int(x[q]), axis=q)
    return psi


def dense_gradient(d, n, gates, x, z):
    """Re <psi|W|psi> and its derivatives in the phases of every T gate, from dense states (adjoint)."""
    psi, snaps = dense(d, n, gates)
    wpsi = dense_weyl(d, psi, x, z)
    wd = psi   # W^dag psi: the shifts are undone first
    for q in range(n):
        if x[q]:
            wd = np.roll(wd, -int(x[q]), axis=q)
        if z[q]:
            wd = _one_site(wd, np.diag(np.exp(-2j * np.pi * z[q] * np.arange(d) / d)), q)
    lam = 0.5 * (wpsi + wd)
    grad = np.zeros((len(snaps), d))
    k = len(snaps)
    for g in reversed(gates):
        if g[0] == "T":
            k -= 1
            ov = (lam.conj() * snaps[k]).sum(axis=tuple(a for a in range(n) if a != g[1]))
            grad[k] = -2.0 * ov.imag
            lam = _one_site(lam, np.diag(np.exp(-1j * np.array(g[2]))), g[1])
        elif g[0] == "SUM":
            for _ in range(d - 1):
                lam = _sum_gate(d, lam, g[1], g[2])
        else:
            lam = _one_site(lam, _gate_matrix(d, g[0]).conj().T, g[1])
    return float(np.vdot(psi, wpsi).real), grad


def parametrised(case, rng):
    """A parametrised circuit and a string whose value and gradient are both well away from 0."""
    d, n = case["d"], case["n"]
    best = (-1.0, None, None, None)
    for _ in range(16):
        gates = named_circuit(d, n, case["layers"], case["t"], rng, parametrised=True)
        x, z, met = evolved_strings(d, n, gates)
        for q in np.argsort(-met, kind="stable")[:4]:
            value, grad = dense_gradient(d, n, gates, x[q], z[q])
            size = min(abs(value), float(np.linalg.norm(grad)))
            if size > best[0]:
                best = (size, gates, x[q], z[q])
        if best[0] > 0.05:
            break
    return best[1:]


def _hash(z):
    z = z + np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def exact(case, seed):
    rng = random.Random(seed)
    d, kind = case["d"], case["kind"]
    if kind == "score":
        th = bond_tensor(d, case["chi_l"], case["chi_r"], seed)
        s2, vn = [], []
        for u in class_unitaries(d):
            t = np.einsum("uv,avb->aub", u, th.reshape(case["chi_l"], d * d, case["chi_r"]))
            p = np.linalg.svd(t.reshape(case["chi_l"] * d, d * case["chi_r"]), compute_uv=False) ** 2
            p = p / p.sum()
            s2.append(-np.log((p * p).sum()))
            vn.append(-(p[p > 0] * np.log(p[p > 0])).sum())
        s2, vn = np.array(s2), np.array(vn)
        if case["via"] == "noalloc":
            return {"s2": s2, "vn": vn, "choice": None}
        return {"s2": s2, "vn": vn if case["score_kind"] != 1 else None, "choice": None, "evaluated": None}
    if kind == "gates":
        n = case["n"]
        gates = named_circuit(d, n, case["layers"], case["t"], rng)
        x, z, _ = evolved_strings(d, n, gates)
        psi, _ = dense(d, n, gates)
        return {"expect": np.array([np.vdot(psi, dense_weyl(d, psi, x[q], z[q])) for q in range(n)]),
                "bond_dims": None}
    if kind == "gradient":
        n = case["n"]
        gates, x, z = parametrised(case, rng)
        value, grad = dense_gradient(d, n, gates, x, z)
        return {"value": value, "grad": grad}
    if kind == "statevector" and not case["disentangle"]:
        # the dense readout fixes the Clifford's free phase by C|0> = P v / |P v|, v a fixed hashed vector and P the
        # projector on C|0>: its phase is that of <C 0|v>
        n = case["n"]
        gates = named_circuit(d, n, case["layers"], case["t"], rng)
        psi, _ = dense(d, n, gates)
        c0, _ = dense(d, n, gates, t_gates=False)
        y = np.arange(d ** n, dtype=np.uint64)
        part = lambda k: (_hash(y * np.uint64(2) + np.uint64(k)) >> np.uint64(11)).astype(np.float64) / 2 ** 53 - 0.5  # noqa: E731,E501
        with np.errstate(over="ignore"):
            v = part(1) + 1j * part(2)
        ph = np.vdot(c0.reshape(-1), v)
        return {"psi": psi.reshape(-1) * (ph / abs(ph))}
    return None
