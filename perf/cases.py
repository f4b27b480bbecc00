"""What this library is used for, as cases that can be timed: batched
contractions of parameterised circuits through `paper_2301_05451_gb300.api`,
from one small circuit to the 20-qubit ansatz with 64 parameter sets, over the
two contraction paths (state sweep, pairwise path) and every kind of result a
program asks for (values, gradients by the adjoint or the shift rule, a
training step, probabilities, amplitudes).

The circuits are the families of `paper_2301_05451_gb300/workloads.py`, written
out here as plain gate lists so that `exact` (64-bit state vectors and a
site-by-site grid contraction in torch / numpy) needs none of the library.

The library computes in float32 and hands values over in float64 slots; the
programs here take them on as float32, the type of their parameters.
"""
import math
import random

import numpy as np
import torch

TWO_PI = 2 * math.pi
DEV = "cuda"


def listed():
    return [
        # one evaluation of the 6-qubit hardware-efficient ansatz (an optimiser's
        # inner step on a small problem): launch latency is all there is
        dict(name="hea6_b1_grad", kind="grad", ansatz="hea", n=6, layers=3, batch=1),
        # one training step of the 12-qubit classifier: forward, loss, backward
        # into the shared weights, through the autograd layer
        dict(name="qnn12_b256_train", kind="train", ansatz="qnn", n=12, layers=4, batch=256),
        # inference of a smaller classifier over a data set of odd size
        dict(name="qnn9_b1001_predict", kind="value", ansatz="qnn", n=9, layers=4, batch=1001),
        # a circuit over the whole gate set, one expectation per qubit and a
        # two-body term, value and gradient (an uneven ansatz search candidate)
        dict(name="random16_b24_grad", kind="grad", ansatz="random", n=16, gates=160, batch=24),
        # an odd-sized ansatz with a handful of parameter sets
        dict(name="ladder17_b5_grad", kind="grad", ansatz="ladder", n=17, layers=6, batch=5),
        # the benchmark's default line: 20 qubits, 64 parameter sets
        dict(name="ladder20_b64_grad", kind="grad", ansatz="ladder", n=20, layers=6, batch=64),
        # the same ansatz, one parameter set, gradient by the shift rule (481 circuits)
        dict(name="ladder20_b1_shift", kind="shift", ansatz="ladder", n=20, layers=6, batch=1),
        # state-vector mode: all 2^20 probabilities of 16 parameter sets from the Neel state
        dict(name="hea20_b16_probs", kind="probs", ansatz="hea", n=20, layers=3, batch=16),
        # twelve uneven circuits (6-12 qubits, 2-6 layers, 8-64 rows) in one launch
        dict(name="multi12_grad", kind="multi", circuits=12, pick=4000),
        # local observable of a 50-qubit grid on its light cone, 32 parameter sets, value and gradient
        dict(name="grid5x10_cone_b32_grad", kind="cone", rows=5, cols=10, layers=4, observed=25, batch=32),
        # one amplitude of a 49-qubit random circuit: sliced hypergraph-partition path
        dict(name="grid7x7_d8_amp", kind="amp", rows=7, cols=7, depth=8, batch=1, method="partition", trials=256,
             target=14),
        # the same along a random-greedy path: few, large pairwise products
        dict(name="grid7x7_d8_amp_greedy", kind="amp", rows=7, cols=7, depth=8, batch=1, method="random_greedy",
             trials=16, target=17),
    ]


def _spread(rng, lo, hi):
    """An integer in [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["grad", "grad", "grad", "train", "value", "shift", "probs", "multi", "cone", "amp"])
    if kind in ("grad", "value"):
        ansatz = rng.choice(["hea", "ladder", "random"] if kind == "grad" else ["hea", "ladder", "random", "qnn"])
        n = rng.randint(4, 20 if kind == "grad" else 18)
        c = dict(kind=kind, ansatz=ansatz, n=n)
        if ansatz == "random":
            c["gates"] = rng.randint(5 * n, 10 * n)
        else:
            c["layers"] = rng.randint(1, 6)
        # at most the state entries of the largest listed case
        c["batch"] = _spread(rng, 1, max(1, min(1500, (32 << 20) >> n)))
        return c
    if kind == "train":
        return dict(kind=kind, ansatz="qnn", n=rng.randint(5, 13), layers=rng.randint(1, 5), batch=_spread(rng, 2, 600))
    if kind == "shift":
        return dict(kind=kind, ansatz=rng.choice(["hea", "ladder"]), n=rng.randint(5, 18), layers=rng.randint(1, 4),
                    batch=rng.randint(1, 3))
    if kind == "probs":
        n = rng.randint(7, 20)
        return dict(kind=kind, ansatz=rng.choice(["hea", "ladder"]), n=n, layers=rng.randint(1, 5),
                    batch=_spread(rng, 1, min(500, (16 << 20) >> n)))
    if kind == "multi":
        return dict(kind=kind, circuits=rng.randint(3, 10), pick=rng.randint(5000, 1 << 20))
    if kind == "cone":
        rows, cols = rng.randint(3, 6), rng.randint(4, 10)
        return dict(kind=kind, rows=rows, cols=cols, layers=rng.randint(2, 4), observed=rng.randrange(rows * cols),
                    batch=_spread(rng, 1, 64))
    return dict(kind="amp", rows=rng.randint(4, 7), cols=rng.randint(4, 7), depth=rng.randint(4, 8),
                batch=rng.randint(1, 4), method="partition", trials=64, target=rng.randint(13, 16))


# ------------------------------------------------------------------ circuits
# A circuit: (n, gates, terms, bits); a gate: (name, qubits, angle sources),
# a source ("p", column) or ("x", feature); a term: (qubits, coefficient,
# group); bits: the amplitude asked for, or None.

class Gates(list):
    def __init__(self):
        self.np = 0

    def rot(self, name, qubits, k=1):
        self.append((name, qubits, tuple(("p", self.np + i) for i in range(k))))
        self.np += k

    def put(self, name, *qubits):
        self.append((name, qubits, ()))


def _ry_rz_cnot(n, layers, ring):
    g = Gates()
    for _ in range(layers):
        for q in range(n):
            g.rot("RY", (q,))
            g.rot("RZ", (q,))
        for q in range(n if ring else n - 1):
            g.put("CNOT", q, (q + 1) % n)
    return g


def _grid_edges(rows, cols):
    """Horizontal even / odd, vertical even / odd."""
    e = [[], [], [], []]
    for r in range(rows):
        for c in range(cols - 1):
            e[c % 2].append((cols * r + c, cols * r + c + 1))
    for r in range(rows - 1):
        for c in range(cols):
            e[2 + r % 2].append((cols * r + c, cols * (r + 1) + c))
    return e


def circuit(c):
    if c["kind"] == "cone":
        n, g, e = c["rows"] * c["cols"], Gates(), _grid_edges(c["rows"], c["cols"])
        for l in range(c["layers"]):
            for a, b in e[l % 4]:
                g.rot("RZZ", (a, b))
            for q in range(n):
                g.rot("RX", (q,))
        return n, g, [((c["observed"],), 1.0, 0)], None
    if c["kind"] == "amp":
        n, g, e = c["rows"] * c["cols"], Gates(), _grid_edges(c["rows"], c["cols"])
        for d in range(c["depth"]):
            for q in range(n):
                g.rot("U3", (q,), 3)
            for a, b in e[d % 4]:
                g.put("CZ", a, b)
        return n, g, [], (0,) * n
    n = c["n"]
    if c["ansatz"] == "hea":
        return n, _ry_rz_cnot(n, c["layers"], True), [((0,), 1.0, 0)], None
    if c["ansatz"] == "ladder":
        return n, _ry_rz_cnot(n, c["layers"], False), [((i, i + 1), 1.0, 0) for i in range(n - 1)], None
    if c["ansatz"] == "qnn":
        g = Gates()
        for q in range(n):
            g.append(("RY", (q,), (("x", q),)))
        for _ in range(c["layers"]):
            for q in range(n):
                g.rot("RX", (q,))
                g.rot("RY", (q,))
                g.rot("RZ", (q,))
            for q in range(n - 1):
                g.put("CZ", q, q + 1)
        return n, g, [((q,), 1.0 / n, 0) for q in range(n)], None
    r, g = random.Random(1000 * n + c["gates"]), Gates()
    for _ in range(c["gates"]):
        name = r.choice(["H", "X", "RX", "RY", "RZ", "U3", "CNOT", "CZ", "RZZ"])
        a, b = r.sample(range(n), 2)
        qubits = (a, b) if name in ("CNOT", "CZ", "RZZ") else (a,)
        k = {"RX": 1, "RY": 1, "RZ": 1, "RZZ": 1, "U3": 3}.get(name, 0)
        g.rot(name, qubits, k) if k else g.put(name, *qubits)
    return n, g, [((q,), 1.0, q) for q in range(n)] + [((0, n - 1), 0.5, n)], None


def _multi(c):
    """The circuits of a multi-circuit launch, as cases of their own."""
    r = np.random.default_rng(c["pick"])
    return [dict(kind="grad", ansatz="ladder", n=int(r.integers(6, 13)), layers=int(r.integers(2, 7)),
                 batch=int(r.choice([8, 16, 32, 64]))) for _ in range(c["circuits"])]


def _rand(seed, *shape):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float32)


def inputs(c, seed):
    """Parameters [batch, P] (or [P] shared), features [batch, F] and targets."""
    if c["kind"] == "multi":
        return [inputs(s, seed * 64 + i)["params"] for i, s in enumerate(_multi(c))]
    n, g, _, _ = circuit(c)
    if c.get("ansatz") == "qnn":  # weights near zero as initialised, features in [0, pi)
        u = _rand(seed, 2, g.np).clamp_min(1e-7)
        w = 0.1 * torch.sqrt(-2 * torch.log(u[0])) * torch.cos(TWO_PI * u[1])
        return dict(params=w, x=math.pi * _rand(seed + 1, c["batch"], n), y=2 * _rand(seed + 2, c["batch"]) - 1)
    return dict(params=TWO_PI * _rand(seed, c["batch"], g.np), x=None)


# ------------------------------------------------------------------ the library's calls

def _spec(c):
    from paper_2301_05451_gb300 import workloads as W
    n, gates, terms, bits = circuit(c)
    s = W.CircuitSpec(n)
    for name, qubits, angles in gates:
        s.add(name, qubits, *angles)
    for qubits, coeff, group in terms:
        s.z(qubits, coeff, group)
    if bits is not None:
        s.amplitude(bits)
    return s


def _neel(n):
    v = torch.zeros(1 << n, dtype=torch.complex64, device=DEV)
    v[int("01" * (n // 2) + "0" * (n % 2), 2)] = 1
    return v


def prepare(c, seed):
    from paper_2301_05451_gb300 import api
    kind, s = c["kind"], {"kind": c["kind"]}
    data = inputs(c, seed)
    if kind == "multi":
        subs = _multi(c)
        s["exec"] = api.MultiExec([api.Circuit(_spec(x)) for x in subs], [x["batch"] for x in subs], grad="adjoint")
        s["params"] = s["exec"].pack([p.cpu() for p in data])
        return s
    s.update(data)
    if kind == "train":
        s["layer"] = api.QuantumLayer(_spec(c), c["batch"], init=data["params"].cpu())
        return s
    C = api.Circuit(_spec(c))
    if kind == "cone":
        net = api.Network(C, "expval", 0, lightcone=True)
        s["exec"] = api.TreeExec(api.Plan(net, method="greedy"), c["batch"], grad="adjoint")
    elif kind == "amp":
        part = c["method"] == "partition"
        net = api.Network(C, "amplitude", 0, hyper=part, split_2q=not part)
        plan = api.Plan(net, method=c["method"], seed=1, temperature=0.3, repeats=c["trials"], target_log2=c["target"])
        s["exec"] = api.TreeExec(plan, c["batch"])
    elif kind == "probs":
        s["exec"] = api.Exec(C, c["batch"], output="probs")
        s["exec"].set_initial_state(_neel(c["n"]))
    else:
        s["exec"] = api.Exec(C, c["batch"], grad={"grad": "adjoint", "shift": "param_shift", "value": "none"}[kind])
    return s


def run(s):
    if s["kind"] == "train":
        layer = s["layer"]
        layer.weight.grad = None
        pred = layer(s["x"]).float().squeeze(-1)
        loss = torch.nn.functional.mse_loss(pred, s["y"])
        loss.backward()
        return {"pred": pred.detach(), "loss": loss.detach(), "grad": layer.weight.grad}
    values, grads = s["exec"].run(s["params"], s.get("x"))
    return {"values": values.float()} if grads is None else {"values": values.float(), "grads": grads}


def work(c):
    """Arithmetic the state sweep cannot do without, per amplitude pair: a real
    rotation 12 flops, a general 2 x 2 gate 28; per amplitude: a phase 6, the
    observable 4.  The adjoint sweep applies every gate to two states and
    takes one dot product per angle (4 per amplitude).  Pairwise paths: the
    state vector of the light cone, or the site-by-site grid contraction.
    Bytes: parameters and features in, values and gradients out."""
    if c["kind"] == "multi":
        ws = [work(x) for x in _multi(c)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    B = c["batch"]
    n, gates, terms, _ = circuit(c)
    P, out = gates.np, 8 * (1 + max([t[2] for t in terms], default=0))
    if c["kind"] == "amp":
        # boundary of `cols` sites, each bond 2^(CZs on the edge); one site at a time
        bond = 2 ** ((c["depth"] + 3) // 4)
        return {"bytes": B * (4.0 * P + 16), "flops": B * 8.0 * n * bond ** (min(c["rows"], c["cols"]) + 1)}
    if c["kind"] == "cone":
        kept, qubits = _cone(gates, terms[0][0])
        gates, n = [gates[i] for i in kept], len(qubits)
    dim, fwd, dots = 2.0 ** n, 0.0, 0.0
    for name, _, angles in gates:
        fwd += {"RX": 6, "RY": 6, "RZ": 6, "RZZ": 6, "U3": 14, "H": 6}.get(name, 0) * dim
        dots += 4 * len(angles) * dim if any(a[0] == "p" for a in angles) else 0
    obs = 4 * dim
    f = {"grad": 3 * fwd + dots + 2 * obs, "cone": 3 * fwd + dots + 2 * obs, "train": 4 * fwd + dots + 3 * obs,
         "value": fwd + obs, "probs": fwd + 3 * dim, "shift": (1 + 2 * P) * (fwd + obs)}[c["kind"]]
    shared = c.get("ansatz") == "qnn"
    by = 4.0 * P * (1 if shared else B) + (4.0 * n * B if shared else 0)
    by += B * (8.0 * dim if c["kind"] == "probs" else out)
    if c["kind"] in ("grad", "cone", "shift", "train"):
        by += 4.0 * P * (1 if shared else B)
    if c["kind"] == "probs":
        by += 8.0 * dim
    return {"bytes": by, "flops": B * f}


# ------------------------------------------------------------------ 64-bit results

def _cone(gates, qubits):
    """Gates in the backward light cone of the qubits, and its qubits."""
    live, kept = set(qubits), []
    for i in range(len(gates) - 1, -1, -1):
        if live & set(gates[i][1]):
            live |= set(gates[i][1])
            kept.append(i)
    return kept[::-1], sorted(live)


def _mat(name, a):
    """2 x 2 tensor [.., 2, 2] of a one-qubit gate at float64 angles a (a list)."""
    if name in ("H", "X"):
        r = math.sqrt(0.5)
        m = [[r, r], [r, -r]] if name == "H" else [[0, 1], [1, 0]]
        return torch.tensor(m, dtype=torch.complex128, device=DEV)
    t = 0.5 * a[0]
    c, s, i = torch.cos(t) + 0j, torch.sin(t) + 0j, 1j
    if name == "RX":
        e = [c, -i * s, -i * s, c]
    elif name == "RY":
        e = [c, -s, s, c]
    elif name == "RZ":
        e = [c - i * s, 0 * c, 0 * c, c + i * s]
    else:  # U3
        p, l = torch.exp(i * a[1]), torch.exp(i * a[2])
        e = [c, -l * s, p * s, p * l * c]
    return torch.stack(e, -1).reshape(e[0].shape + (2, 2))


def _dmat(name, a, j):
    """Derivative of _mat with respect to angle j."""
    if j == 0:  # every matrix depends on angle 0 through cos, sin of its half
        shifted = [a[0] + math.pi] + list(a[1:])
        return 0.5 * _mat(name, shifted)
    m = _mat(name, a).clone()
    m[..., 0, :] *= 0 if j == 1 else 1
    m[..., :, 0] *= 0 if j == 2 else 1
    return 1j * m


def _one(psi, n, q, m):
    """m ([2, 2] or [B, 2, 2]) on qubit q (0 = most significant bit) of psi [B, 2^n]."""
    v = psi.view(psi.shape[0], 1 << q, 2, -1)
    m = m.reshape(-1, 2, 2, 1, 1).expand(psi.shape[0], 2, 2, 1, 1)
    return torch.stack([m[:, 0, 0] * v[:, :, 0] + m[:, 0, 1] * v[:, :, 1],
                        m[:, 1, 0] * v[:, :, 0] + m[:, 1, 1] * v[:, :, 1]], 2).reshape(psi.shape)


def _sign(n, qubits):
    """(-1)^(parity of the qubits' bits) over the basis."""
    x = torch.arange(1 << n, device=DEV)
    s = torch.zeros_like(x)
    for q in qubits:
        s ^= (x >> (n - 1 - q)) & 1
    return 1.0 - 2.0 * s.double()


def _gate(psi, n, name, qubits, a, dag=False):
    if name == "CNOT":
        x = torch.arange(1 << n, device=DEV)
        return psi[:, x ^ (((x >> (n - 1 - qubits[0])) & 1) << (n - 1 - qubits[1]))]
    if name == "CZ":
        x = torch.arange(1 << n, device=DEV)
        return psi * (1.0 - 2.0 * ((x >> (n - 1 - qubits[0])) & (x >> (n - 1 - qubits[1])) & 1).double())
    if name == "RZZ":
        t = (0.5j if dag else -0.5j) * a[0]
        return psi * torch.exp(t.reshape(-1, 1) * _sign(n, qubits))
    m = _mat(name, a)
    return _one(psi, n, qubits[0], m.conj().transpose(-1, -2) if dag else m)


def _sweep(n, gates, terms, P, params, x, grad, psi=None, weight=None):
    """Values [B, groups], gradients [B, P] of sum_g weight_g value_g, final states."""
    rows = max(params.shape[0], 1 if x is None else x.shape[0])
    ang = [[(params[:, k] if s == "p" else x[:, k]) for s, k in angles] for _, _, angles in gates]
    if psi is None:
        psi = torch.zeros(rows, 1 << n, dtype=torch.complex128, device=DEV)
        psi[:, 0] = 1
    for (name, qubits, _), a in zip(gates, ang):
        psi = _gate(psi, n, name, qubits, a)
    groups = 1 + max([t[2] for t in terms], default=-1)
    diag = torch.zeros(groups, 1 << n, dtype=torch.float64, device=DEV)
    for qubits, coeff, g in terms:
        diag[g] += coeff * _sign(n, qubits)
    values = (psi.abs() ** 2) @ diag.T
    if not grad:
        return values, None, psi
    w = torch.ones(rows, groups, dtype=torch.float64, device=DEV) if weight is None else weight(values)
    lam = psi * (w @ diag)
    grads = torch.zeros(rows, P, dtype=torch.float64, device=DEV)
    for (name, qubits, angles), a in zip(reversed(gates), reversed(ang)):
        if name == "RZZ" or name == "RZ":  # d/dt: -i/2 Z (x Z)
            grads[:, angles[0][1]] += ((lam.conj() * psi).imag * _sign(n, qubits)).sum(1)
            psi, lam = _gate(psi, n, name, qubits, a, True), _gate(lam, n, name, qubits, a, True)
            continue
        psi = _gate(psi, n, name, qubits, a, True)
        for j, (s, k) in enumerate(angles):
            if s == "p":
                d = _one(psi, n, qubits[0], _dmat(name, a, j))
                grads[:, k] += 2 * (lam.real * d.real + lam.imag * d.imag).sum(1)
        lam = _gate(lam, n, name, qubits, a, True)
    return values, grads, psi


def _grid_amplitude(c, gates, params):
    """<0|U|0> of one parameter row: the sites' tensors (one bond bit per CZ on
    an edge) contracted row by row with a boundary over the columns."""
    rows, cols = c["rows"], c["cols"]
    bonds = [[] for _ in range(rows * cols)]  # the other site of each bond, in time order
    acc = [np.array([1, 0], np.complex128) for _ in range(rows * cols)]  # [2, bond bits ...]
    for name, qubits, angles in gates:
        if name == "U3":
            t, p, l = (float(params[k]) for _, k in angles)
            co, si = math.cos(t / 2), math.sin(t / 2)
            m = np.array([[co, -np.exp(1j * l) * si], [np.exp(1j * p) * si, np.exp(1j * (p + l)) * co]])
            acc[qubits[0]] = np.tensordot(m, acc[qubits[0]], (1, 0))
        else:  # CZ = sum_s |s><s| (x) Z^s: the first qubit copies s, the second applies Z^s
            a, b = qubits
            acc[a] = np.stack([acc[a] * np.array([1, 0]).reshape((2,) + (1,) * (acc[a].ndim - 1)),
                               acc[a] * np.array([0, 1]).reshape((2,) + (1,) * (acc[a].ndim - 1))], -1)
            acc[b] = np.stack([acc[b], acc[b] * np.array([1, -1]).reshape((2,) + (1,) * (acc[b].ndim - 1))], -1)
            bonds[a].append(b)
            bonds[b].append(a)
    # tensors [up, left, down, right], bonds of one edge grouped in time order
    bound, dims = np.ones((1,), np.complex128), [1] * cols  # boundary over the columns' down bonds
    for r in range(rows):
        cur = bound.reshape(dims + [1])  # ..., left bond
        ndims = []
        for k in range(cols):
            s = r * cols + k
            t = acc[s][0]
            want = [s - cols, s - 1, s + cols, s + 1]
            order = [[i for i, o in enumerate(bonds[s]) if o == w] for w in want]
            if k == 0:
                order[1] = []
            if k == cols - 1:
                order[3] = []
            t = np.transpose(t, sum(order, [])) if t.ndim else t
            t = t.reshape([2 ** len(o) for o in order])
            # cur axes: remaining up bonds (k.. cols-1), finished down bonds (0..k-1), left
            cur = np.tensordot(cur, t, ([0, cur.ndim - 1], [0, 1]))
            ndims.append(t.shape[2])
        bound, dims = cur.reshape(-1), ndims
    return complex(bound.reshape(-1)[0])


def exact(c, seed):
    data = inputs(c, seed)
    if c["kind"] == "multi":
        vs, gs = [], []
        for s, p in zip(_multi(c), data):
            n, gates, terms, _ = circuit(s)
            v, g, _ = _sweep(n, gates, terms, gates.np, p.double(), None, True)
            vs.append(v.reshape(-1))
            gs.append(g.reshape(-1))
        return {"values": torch.cat(vs), "grads": torch.cat(gs)}
    n, gates, terms, _ = circuit(c)
    p = data["params"].double()
    if c["kind"] == "amp":
        a = [_grid_amplitude(c, gates, row) for row in p.cpu().numpy()]
        return {"values": torch.tensor([[z.real, z.imag] for z in a], dtype=torch.float64)}
    if c["kind"] == "cone":
        kept, qubits = _cone(gates, terms[0][0])
        at = {q: i for i, q in enumerate(qubits)}
        sub = [(gates[i][0], tuple(at[q] for q in gates[i][1]), gates[i][2]) for i in kept]
        v, g, _ = _sweep(len(qubits), sub, [(tuple(at[q] for q in terms[0][0]), 1.0, 0)], gates.np, p, None, True)
        return {"values": v, "grads": g}
    if c["kind"] == "probs":
        _, _, psi = _sweep(n, gates, [], gates.np, p, None, False,
                           psi=_neel(n).to(torch.complex128).expand(c["batch"], -1).clone())
        return {"values": psi.real ** 2 + psi.imag ** 2}
    x = None if data["x"] is None else data["x"].double()
    p2 = p if p.dim() == 2 else p[None, :].expand(c["batch"], -1)
    if c["kind"] == "train":
        y = data["y"].double()
        v, g, _ = _sweep(n, gates, terms, gates.np, p2, x, True, weight=lambda v: 2 * (v - y[:, None]) / len(y))
        v = v.squeeze(-1)
        return {"pred": v, "loss": ((v - y) ** 2).mean(), "grad": g.sum(0)}
    v, g, _ = _sweep(n, gates, terms, gates.np, p2, x, c["kind"] != "value")
    return {"values": v} if g is None else {"values": v, "grads": g}
