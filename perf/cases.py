"""The work that a user of this framework has it do, as cases that can be timed.

Kinds of case, each through the public binding (paper_2211_17028_gb300.nqs):

  fidelity  NoisyCircuit.fidelity: A(l) of one noisy circuit, from the smallest
            calls (a few qubits, launches count) through the widths that the
            precompiled sweep kernels serve up to the widths that get kernels
            of their own (26 qubits and more)
  general   the same call on a circuit with two-qubit noise channels
  batch     nqs_batch_fidelity: many circuits of mixed widths in one call
  sets      nqs_eval_sets: the weights of chosen site triples, the inner step
            of an importance-sampled level-3 sum
  mlp       nqs_mlp_loss_grad: loss and gradient of one batch of the proposal
            network (forward and backward, bf16 weights)
  reduced   nqs_reduced_matrix: the reduced 2x2 matrix of two states

The circuits are the structures of this repository's own workloads: lines and
grids of U3 layers with alternating CZ patterns, QAOA MaxCut on 3-regular
graphs, amplitude- and phase-damping and depolarizing noises at rates between
1e-4 and 1e-2.  What a case is (widths, gate and noise positions) follows from
its fields; angles, rates, bit strings, states and weights follow from the
seed.  The one exception are the circuits of 26 qubits and more: their kernels
are compiled for the circuit, so a program keeps the circuit and changes the
input state; there the seed gives the state alone.

Fidelities come back as the numbers of the result record.  Sweeps run in
complex64; where many results are put into one array, it is an array of
single precision, which is what these results carry.
"""

import math
import random

import numpy as np
import torch

from paper_2211_17028_gb300 import nqs

TWO_PI = 2.0 * math.pi
JIT_QUBITS = 26          # from here on the library compiles kernels for a circuit


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call in use: six qubits, every term up to level 4
        {"name": "line6_l4", "kind": "fidelity", "family": "line", "n": 6, "depth": 8, "noises": 4,
         "channel": "depol", "level": 4, "psi": "basis", "v": "basis", "circuit": 1},
        # a small odd width with a ragged number of noises, v = U|psi>
        {"name": "line13_l2", "kind": "fidelity", "family": "line", "n": 13, "depth": 14, "noises": 11,
         "channel": "mixed", "level": 2, "psi": "basis", "v": "ideal", "circuit": 2},
        # dense input and test states, a deeper level
        {"name": "grid16_l3", "kind": "fidelity", "family": "grid", "n": 16, "depth": 10, "noises": 8,
         "channel": "adpd", "level": 3, "psi": "dense", "v": "dense", "circuit": 3},
        # the usual study: 4x5 grid, 20 damping noises, level 2, a bit string
        {"name": "grid20_l2", "kind": "fidelity", "family": "grid", "n": 20, "depth": 16, "noises": 20,
         "channel": "adpd", "level": 2, "psi": "basis", "v": "basis", "circuit": 4},
        # QAOA at the widest circuits of a batch study
        {"name": "qaoa24_l2", "kind": "fidelity", "family": "qaoa", "n": 24, "depth": 4, "noises": 20,
         "channel": "depol", "level": 2, "psi": "basis", "v": "ideal", "circuit": 5},
        # level 1 (often enough, at any width): 40 noises, two sweeps
        {"name": "grid25_l1", "kind": "fidelity", "family": "grid", "n": 25, "depth": 12, "noises": 40,
         "channel": "mixed", "level": 1, "psi": "basis", "v": "basis", "circuit": 6},
        # the headline QAOA study, at the width whose states fit three times
        {"name": "qaoa28_l2", "kind": "fidelity", "family": "qaoa", "n": 28, "depth": 4, "noises": 20,
         "channel": "depol", "level": 2, "psi": "basis", "v": "ideal", "circuit": 7},
        # two-qubit depolarizing noises after two-qubit gates
        {"name": "general12_l2", "kind": "general", "family": "line", "n": 12, "depth": 6, "noises": 4,
         "channel": "depol2", "level": 2, "psi": "basis", "v": "ideal", "circuit": 8},
        # a batch of unlike circuits in one call
        {"name": "batch32", "kind": "batch", "count": 32, "n_lo": 12, "n_hi": 21, "noises_hi": 30, "circuit": 9},
        # site triples of the 4x5 grid with 200 noises
        {"name": "sets20", "kind": "sets", "n": 20, "depth": 24, "noises": 200, "sets": 40, "circuit": 10},
        # one training batch of the proposal network, 8 -> 256 x 3 -> 1
        {"name": "mlp1024", "kind": "mlp", "batch": 1024},
        # the reduced matrix of two wide states
        {"name": "reduced28", "kind": "reduced", "n": 28, "qubit": 11},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= 0.2 * most:
            return c


def _draw(rng):
    kind = rng.choice(("fidelity",) * 6 + ("general", "batch", "sets", "mlp", "reduced"))
    c = {"kind": kind, "circuit": rng.randrange(1, 1 << 20)}
    if kind == "fidelity":
        c["family"] = rng.choice(("line", "grid", "qaoa"))
        n = rng.randint(4, 27)
        if c["family"] == "qaoa":
            n = max(4, n - n % 2)
        if c["family"] == "grid" and not _grid_dims(n):
            c["family"] = "line"
        level = rng.choice((1, 1, 2, 2, 2, 3))
        c.update(n=n, depth=rng.randint(2, 4) if c["family"] == "qaoa" else rng.randint(6, 24),
                 noises=rng.randint(4, 12 if level == 3 or n > 24 else 40),
                 channel=rng.choice(("depol", "adpd", "mixed")), level=level,
                 psi=rng.choice(("basis", "basis", "dense")), v=rng.choice(("basis", "ideal", "dense")))
    elif kind == "general":
        c.update(family="line", n=rng.randint(4, 16), depth=rng.randint(3, 8), noises=rng.randint(2, 5),
                 channel="depol2", level=rng.choice((1, 2)), psi="basis", v=rng.choice(("basis", "ideal")))
    elif kind == "batch":
        lo = rng.randint(12, 16)
        c.update(count=_log_int(rng, 4, 48), n_lo=lo, n_hi=rng.randint(lo, 22), noises_hi=rng.randint(6, 36))
    elif kind == "sets":
        n = rng.randint(12, 20)
        c.update(n=n, depth=rng.randint(12, 24), noises=rng.randint(30, 200), sets=_log_int(rng, 4, 40))
    elif kind == "mlp":
        c.update(batch=_log_int(rng, 50, 8192))
    else:
        n = rng.randint(8, 28)
        c.update(n=n, qubit=rng.randrange(n))
    return c


# ------------------------------------------------------- circuits and channels

def _grid_dims(n):
    for r in range(int(math.isqrt(n)), 1, -1):
        if n % r == 0:
            return r, n // r
    return None


def _three_regular(rng, n):
    while True:
        stubs = [v for v in range(n) for _ in range(3)]
        rng.shuffle(stubs)
        edges = {(min(a, b), max(a, b)) for a, b in zip(stubs[::2], stubs[1::2])}
        if len(edges) == 3 * n // 2 and all(a != b for a, b in edges):
            return sorted(edges)


def _gates(place, values, family, n, depth):
    """[(name, qubits, params)]: positions from `place`, angles from `values`."""
    gates = []
    if family == "qaoa":
        edges = _three_regular(place, n)
        gates += [("h", (q,), ()) for q in range(n)]
        for _ in range(depth):
            gamma, beta = values.uniform(0, math.pi), values.uniform(0, math.pi)
            for a, b in edges:
                gates += [("cx", (a, b), ()), ("rz", (b,), (2 * gamma,)), ("cx", (a, b), ())]
            gates += [("rx", (q,), (2 * beta,)) for q in range(n)]
        return gates
    rows, cols = _grid_dims(n) if family == "grid" else (1, n)
    for layer in range(depth):
        gates += [("u3", (q,), tuple(values.uniform(0, TWO_PI) for _ in range(3))) for q in range(n)]
        if family == "line":
            pairs = [(q, q + 1) for q in range(layer % 2, n - 1, 2)]
        elif layer % 4 < 2:
            pairs = [(r * cols + c, r * cols + c + 1) for r in range(rows) for c in range(layer % 2, cols - 1, 2)]
        else:
            pairs = [(r * cols + c, (r + 1) * cols + c) for r in range(layer % 2, rows - 1, 2) for c in range(cols)]
        gates += [("cz", p, ()) for p in pairs]
    return gates


_I = np.eye(2, dtype=np.complex128)
_PAULIS = [_I, np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]]), np.diag([1.0 + 0j, -1.0])]


def _damping(gamma):
    return [np.diag([1.0 + 0j, math.sqrt(1 - gamma)]), np.array([[0, math.sqrt(gamma)], [0, 0]], complex)]


def _dephasing(lam):
    return [np.diag([1.0 + 0j, math.sqrt(1 - lam)]), np.diag([0j, math.sqrt(lam)])]


def _kraus(place, values, channel):
    rate = math.exp(values.uniform(math.log(1e-4), math.log(1e-2)))
    if channel == "mixed":
        channel = place.choice(("ad", "pd", "depol"))
    if channel == "ad":
        return _damping(rate)
    if channel == "pd":
        return _dephasing(rate)
    if channel == "adpd":
        return [m for m in (a @ b for a in _dephasing(rate) for b in _damping(rate)) if m.any()]
    if channel == "depol":
        return [math.sqrt(1 - rate) * _I] + [math.sqrt(rate / 3) * p for p in _PAULIS[1:]]
    pairs = [np.kron(p, q) for p in _PAULIS for q in _PAULIS]
    return [math.sqrt(1 - rate) * pairs[0]] + [math.sqrt(rate / 15) * p for p in pairs[1:]]


def _circuit(place, values, family, n, depth, noises, channel):
    """(n, gates, [(after gate, qubits, Kraus operators)])"""
    gates = _gates(place, values, family, n, depth)
    spots = [g for g, x in enumerate(gates) if channel != "depol2" or len(x[1]) == 2]
    sites = []
    for g in sorted(place.sample(spots, min(noises, len(spots)))):
        qs = gates[g][1] if channel == "depol2" else (place.choice(gates[g][1]),)
        sites.append((g, qs, _kraus(place, values, channel)))
    return n, gates, sites


def _text(circuit):
    n, gates, sites = circuit
    lines = ["nqs-ir 1", "qubits %d" % n]
    for name, qs, params in gates:
        lines.append("gate %s %s" % (name, " ".join([str(q) for q in qs] + [repr(float(p)) for p in params])))
    for g, qs, kraus in sites:
        nums = " ".join(repr(float(x)) for k in kraus for x in np.ascontiguousarray(k).view(np.float64).reshape(-1))
        lines.append("%s %d %s %d %s" % ("noise2" if len(qs) == 2 else "noise", g, " ".join(map(str, qs)),
                                         len(kraus), nums))
    return "\n".join(lines) + "\n"


def _circuit_of(case, seed):
    """The case's circuit and the generator of what is left to draw from the seed."""
    place, values = random.Random(case["circuit"]), random.Random(seed)
    if case["kind"] == "sets":
        fields = ("grid" if _grid_dims(case["n"]) else "line", case["n"], case["depth"], case["noises"], "mixed")
    else:
        fields = tuple(case[k] for k in ("family", "n", "depth", "noises", "channel"))
    own = random.Random(case["circuit"] + 1) if case["n"] >= JIT_QUBITS else values
    return _circuit(place, own, *fields), values


def _batch_of(case, seed):
    """[(circuit, level)] of a batch"""
    place, values = random.Random(case["circuit"]), random.Random(seed)
    out = []
    for _ in range(case["count"]):
        n = place.randint(case["n_lo"], case["n_hi"])
        family = "grid" if _grid_dims(n) and place.random() < 0.5 else "line"
        c = _circuit(place, values, family, n, place.randint(10, 30), place.randint(5, case["noises_hi"]), "mixed")
        out.append((c, place.randint(1, 2)))
    return out


def _dense(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(1 << n, 2, device="cuda", generator=g)
    return torch.view_as_complex(x / x.norm())


def _states(case, seed, values):
    """What psi and v are: bits of a basis state, a dense vector, or None for U|psi>."""
    psi = values.getrandbits(case["n"]) if case["psi"] == "basis" else _dense(case["n"], 2 * seed)
    v = {"basis": lambda: values.getrandbits(case["n"]), "ideal": lambda: None,
         "dense": lambda: _dense(case["n"], 2 * seed + 1)}[case["v"]]()
    return psi, v


def _descriptor(x):
    return nqs.ideal() if x is None else nqs.basis(x) if isinstance(x, int) else nqs.dense(x)


def _site_sets(case, seed):
    values = random.Random(seed + 1)
    sets = {tuple(sorted(values.sample(range(case["noises"]), 3))) for _ in range(case["sets"])}
    return np.array(sorted(sets), dtype=np.int32)


MLP_DIMS = (8, 256, 256, 256, 1)


def _mlp_inputs(case, seed):
    rng = np.random.RandomState(seed % (1 << 31))
    params = [p for a, b in zip(MLP_DIMS, MLP_DIMS[1:])
              for p in (rng.uniform(-1, 1, (b, a)) / math.sqrt(a), rng.uniform(-0.1, 0.1, b))]
    x = rng.standard_normal((case["batch"], MLP_DIMS[0])).astype(np.float32)
    y = (x[:, 2] + x[:, 6] - 10 + rng.standard_normal(case["batch"])).astype(np.float32)
    return [p.astype(np.float32) for p in params], x, y


# ------------------------------------------------------------ prepare and run

class _Mlp:
    def __init__(self, params):
        self.m = nqs.nqs_mlp_create(MLP_DIMS[0], MLP_DIMS[1], len(MLP_DIMS) - 2, 0)
        nqs.nqs_mlp_set_params(self.m, np.concatenate([p.reshape(-1) for p in params]))

    def __del__(self):
        nqs.nqs_mlp_destroy(self.m)


def prepare(case, seed):
    nqs.use_torch_allocator()
    kind = case["kind"]
    state = {"kind": kind}
    if kind in ("fidelity", "general"):
        circuit, values = _circuit_of(case, seed)
        psi, v = _states(case, seed, values)
        state.update(circuit=nqs.NoisyCircuit(_text(circuit)), keep=(psi, v), psi=_descriptor(psi),
                     v=_descriptor(v), level=case["level"])
    elif kind == "batch":
        batch = _batch_of(case, seed)
        state.update(circuits=[nqs.NoisyCircuit(_text(c)) for c, _ in batch], levels=[l for _, l in batch],
                     psis=[nqs.basis(0) for _ in batch], vs=[nqs.ideal() for _ in batch])
        state["handles"] = [c.h for c in state["circuits"]]
    elif kind == "sets":
        circuit, _ = _circuit_of(case, seed)
        state.update(circuit=nqs.NoisyCircuit(_text(circuit)), sets=_site_sets(case, seed))
        nqs.nqs_prepare_sets(state["circuit"].h, nqs.basis(0), nqs.ideal())
    elif kind == "mlp":
        params, x, y = _mlp_inputs(case, seed)
        state.update(mlp=_Mlp(params), x=torch.from_numpy(x).cuda(), y=torch.from_numpy(y).cuda())
    else:
        n = case["n"]
        bytes_ = nqs.nqs_reduced_matrix_scratch_bytes(n)
        state.update(phi=_dense(n, 2 * seed), chi=_dense(n, 2 * seed + 1), n=n, qubit=case["qubit"],
                     out=torch.zeros(8, dtype=torch.float64, device="cuda"), bytes=bytes_,
                     scratch=torch.empty(bytes_, dtype=torch.uint8, device="cuda"))
    return state


def run(s):
    kind = s["kind"]
    if kind in ("fidelity", "general"):
        return s["circuit"].fidelity(s["psi"], s["v"], s["level"])
    if kind == "batch":
        rs = nqs.nqs_batch_fidelity(s["handles"], s["psis"], s["vs"], s["levels"])
        return {"F": torch.tensor([r.F for r in rs]), "T": torch.tensor([list(r.T[:3]) for r in rs]),
                "n_terms": torch.tensor([int(r.n_terms) for r in rs]), "status": torch.tensor([r.status for r in rs])}
    if kind == "sets":
        return torch.tensor(nqs.nqs_eval_sets(s["circuit"].h, s["sets"]), dtype=torch.float32)
    if kind == "mlp":
        loss, grad = nqs.nqs_mlp_loss_grad(s["mlp"].m, s["x"], s["y"])
        return {"loss": loss, "grad": grad}
    nqs.nqs_reduced_matrix(s["phi"], s["chi"], s["n"], s["qubit"], s["out"], s["scratch"], s["bytes"])
    return s["out"]


# ----------------------------------------------------------------------- work

def _expansion_work(n, gates, N, level, ideal, rest):
    """Sweeps of one expansion.  Every dense gate acts once on every state swept:
    the input state, the test state (and U|psi>), and each state with d < level
    insertions, which starts on average after d/(d+1) of the circuit; it is a
    2x2 product, 14 flops an amplitude (diagonal gates can be folded into
    these).  Memory: every checkpoint of the test state written once, and read
    once for each group of states that is reduced against it."""
    N = max(N, 1)
    level = min(level, N)
    sweeps = 2.0 + (1.0 if ideal else 0.0)
    reads = 2.0 * N
    for d in range(1, level):
        sweeps += math.comb(N, d) * rest ** d / (d + 1)
        reads += math.comb(N, d + 1) * rest ** (d - 1)
    return {"bytes": 8.0 * 2 ** n * reads, "flops": 14.0 * 2 ** n * gates * sweeps}


def _dense_gates(c):
    return c["n"] * (c["depth"] + (1 if c["family"] == "qaoa" else 0))


def work(case):
    kind = case["kind"]
    if kind in ("fidelity", "general"):
        return _expansion_work(case["n"], _dense_gates(case), case["noises"], case["level"], case["v"] == "ideal",
                               15 if kind == "general" else 3)
    if kind == "batch":
        parts = [_expansion_work(c[0], sum(len(g[1]) == 1 for g in c[1]), len(c[2]), level, True, 3) for c, level in _batch_of(case, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "sets":
        # three states from the first site to the second, nine to the third: a
        # quarter of the circuit each; two checkpoints read
        amps = 2.0 ** case["n"] * case["sets"]
        return {"bytes": 16.0 * amps, "flops": 14.0 * amps * case["n"] * case["depth"] * 0.25 * 12}
    if kind == "mlp":
        weights = sum(a * b for a, b in zip(MLP_DIMS, MLP_DIMS[1:]))
        return {"bytes": 4.0 * case["batch"] * (MLP_DIMS[0] + 1) + 8.0 * weights, "flops": 6.0 * weights * case["batch"]}
    return {"bytes": 16.0 * 2 ** case["n"], "flops": 32.0 * 2 ** case["n"] / 2}


def _cost(case):
    w = work(case)
    return max(w["bytes"] / 6e12, w["flops"] / 4e13)


# ------------------------------------------------------- the same in 64 bits

def _gate_matrix(name, p):
    if name == "u3":
        t, phi, lam = p
        return np.array([[math.cos(t / 2), -np.exp(1j * lam) * math.sin(t / 2)],
                         [np.exp(1j * phi) * math.sin(t / 2), np.exp(1j * (phi + lam)) * math.cos(t / 2)]])
    if name == "h":
        return np.array([[1, 1], [1, -1]], complex) / math.sqrt(2)
    if name == "rx":
        return math.cos(p[0] / 2) * _I - 1j * math.sin(p[0] / 2) * _PAULIS[1]
    return np.diag([np.exp(-0.5j * p[0]), np.exp(0.5j * p[0])])


def _apply(x, qs, m):
    """m on the qubits qs of the states x [states, 2^n], in place where it can be"""
    states, dim = x.shape
    if len(qs) == 1:
        y = x.view(states, dim >> (qs[0] + 1), 2, 1 << qs[0])
        if m[0, 1] == 0 and m[1, 0] == 0:
            for b in range(2):
                if m[b, b] != 1:
                    y[:, :, b] *= complex(m[b, b])
            return x
        a, b = y[:, :, 0].clone(), y[:, :, 1].clone()
        for r in range(2):
            torch.add(complex(m[r, 0]) * a, b, alpha=complex(m[r, 1]), out=y[:, :, r])
        return x
    hi, lo = max(qs), min(qs)
    y = x.view(states, dim >> (hi + 1), 2, 1 << (hi - lo - 1), 2, 1 << lo)
    part = lambda i: y[:, :, i >> 1, :, i & 1] if qs[0] == hi else y[:, :, i & 1, :, i >> 1]  # noqa: E731
    if isinstance(m, str):
        if m == "cz":
            part(3).neg_()
        else:
            a = part(2).clone()
            part(2).copy_(part(3))
            part(3).copy_(a)
        return x
    old = [part(i).clone() for i in range(4)]
    for r in range(4):
        acc = complex(m[r, 0]) * old[0]
        for c in range(1, 4):
            if m[r, c] != 0:
                acc = acc + complex(m[r, c]) * old[c]
        part(r).copy_(acc)
    return x


class _Reference:
    """The level-l expansion (Sec. IV, Algorithm 1) in complex128."""

    def __init__(self, circuit, psi, v):
        self.n, gates, sites = circuit
        self.ops, self.K = [], []
        at = 0
        for g in range(len(gates)):
            name, qs, p = gates[g]
            self.ops.append((qs, name if len(qs) == 2 else _gate_matrix(name, p), -1))
            while at < len(sites) and sites[at][0] == g:
                _, qs, kraus = sites[at]
                vecs = np.array([k.reshape(-1) for k in kraus]).T
                d, u = np.linalg.eigh(vecs @ vecs.conj().T)
                order = np.argsort(-d)
                self.K.append([math.sqrt(max(d[i], 0.0)) * u[:, i].reshape(kraus[0].shape) for i in order])
                self.ops.append((qs, self.K[-1][0], at))
                at += 1
        self.psi = self.vector(psi)
        if v is None:
            self.v = self.psi.clone()
            for qs, m, s in self.ops:
                if s < 0:
                    _apply(self.v, qs, m)
        else:
            self.v = self.vector(v)

    def vector(self, x):
        if isinstance(x, int):
            out = torch.zeros(1, 1 << self.n, dtype=torch.complex128, device="cuda")
            out[0, x] = 1
            return out
        return x.to(torch.complex128).reshape(1, -1).clone()

    def backward(self):
        phi, x = {}, self.v.clone()
        for qs, m, s in reversed(self.ops):
            if s >= 0:
                phi[s] = x.clone()
            _apply(x, qs, m if isinstance(m, str) else m.conj().T)
        return phi

    def reduced(self, phi, x, qs):
        """R[state][a, b] = sum over the other qubits of conj(phi[.. a ..]) x[.. b ..]"""
        dim = 1 << self.n
        if len(qs) == 1:
            f = phi.view(dim >> (qs[0] + 1), 2, 1 << qs[0])
            y = x.view(-1, dim >> (qs[0] + 1), 2, 1 << qs[0])
            parts, of = [f[:, a] for a in range(2)], [y[:, :, b] for b in range(2)]
        else:
            hi, lo = max(qs), min(qs)
            f = phi.view(dim >> (hi + 1), 2, 1 << (hi - lo - 1), 2, 1 << lo)
            y = x.view(-1, *f.shape)
            at = [(i >> 1, i & 1) if qs[0] == hi else (i & 1, i >> 1) for i in range(4)]
            parts, of = [f[:, i, :, j] for i, j in at], [y[:, :, i, :, j] for i, j in at]
        return torch.stack([torch.stack([(p.conj() * o).flatten(1).sum(1) for o in of], 1) for p in parts], 1)

    def amps(self, phi, x, s, qs, which):
        """<phi_s| K_i x> for the factors `which`: [states, factors]"""
        K = torch.tensor(np.array([self.K[s][i] for i in which]), device="cuda")
        return torch.einsum("iab,sab->si", K, self.reduced(phi, x, qs))

    def spawn(self, x, s, qs):
        return torch.cat([_apply(x.clone(), qs, self.K[s][i]) for i in range(1, len(self.K[s]))])

    def levels(self, level):
        """T_0 .. T_level"""
        phi = self.backward()
        T = [0.0] * (level + 1)
        last = max((i for i, o in enumerate(self.ops) if o[2] >= 0), default=-1)

        def expand(x, at, depth):
            for i in range(at, last + 1):
                qs, m, s = self.ops[i]
                if s >= 0 and depth < level:
                    a = self.amps(phi[s], x, s, qs, range(1, len(self.K[s])))
                    T[depth + 1] += a.abs().square().sum()
                    if depth + 1 < level:
                        expand(self.spawn(x, s, qs), i + 1, depth + 1)
                if s >= 0 and depth == 0 and i == last:
                    T[0] = self.amps(phi[s], x, s, qs, [0]).abs().square().sum()
                _apply(x, qs, m)

        expand(self.psi.clone(), 0, 0)
        return [float(t) for t in T]

    def weights(self, sets):
        """W(S) of site triples: the sum of the term values over their factors"""
        phi, chi, where = self.backward(), {}, {}
        x = self.psi.clone()
        for i, (qs, m, s) in enumerate(self.ops):
            if s >= 0:
                chi[s], where[s] = x.clone(), i
            _apply(x, qs, m)
        out = []
        for a, b, c in sets.tolist():
            x = self.spawn(chi[a].clone(), a, self.ops[where[a]][0])
            for qs, m, s in self.ops[where[a] + 1:where[c]]:
                x = self.spawn(x, s, qs) if s == b else _apply(x, qs, m)
            qs = self.ops[where[c]][0]
            out.append(float(self.amps(phi[c], x, c, qs, range(1, 4)).abs().square().sum()))
        return torch.tensor(out, dtype=torch.float64)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fidelity", "general"):
        circuit, values = _circuit_of(case, seed)
        psi, v = _states(case, seed, values)
        # level 2 of a wide circuit takes minutes in 64 bits: its levels 0 and 1 alone
        level = min(case["level"], case["noises"])
        done = level if _cost(case) < 0.03 else min(level, 1)
        T = _Reference(circuit, psi, v).levels(done)
        return {"F": math.fsum(T) if done == level else None, "T": T + [None] * (level - done),
                "imag_residual": None, "n_terms": None, "bound": None, "level": None, "status": None}
    if kind == "batch":
        if _cost(case) > 0.06:
            return None
        Ts = [_Reference(c, 0, None).levels(level) for c, level in _batch_of(case, seed)]
        return {"F": torch.tensor([math.fsum(T) for T in Ts], dtype=torch.float64),
                "T": torch.tensor([T + [0.0] * (3 - len(T)) for T in Ts], dtype=torch.float64),
                "n_terms": None, "status": None}
    if kind == "sets":
        circuit, _ = _circuit_of(case, seed)
        return _Reference(circuit, 0, None).weights(_site_sets(case, seed))
    if kind == "mlp":
        params, x, y = _mlp_inputs(case, seed)
        p = [torch.from_numpy(a) for a in params]
        # the products use the weights in bf16; biases and data in fp32
        p = [(a.bfloat16() if i % 2 == 0 else a).double().cuda().requires_grad_() for i, a in enumerate(p)]
        h = torch.from_numpy(x).double().cuda()
        for i in range(0, len(p), 2):
            h = h @ p[i].T + p[i + 1]
            h = torch.relu(h) if i + 2 < len(p) else h
        loss = (h[:, 0] - torch.from_numpy(y).double().cuda()).square().mean()
        loss.backward()
        return {"loss": float(loss.detach()), "grad": torch.cat([a.grad.reshape(-1) for a in p])}
    n, q = case["n"], case["qubit"]
    f, x = (_dense(n, 2 * seed + k).view(1 << (n - 1 - q), 2, 1 << q) for k in range(2))
    total = torch.zeros(4, dtype=torch.complex128, device="cuda")
    step = max(1, (1 << 24) >> q)
    for at in range(0, f.shape[0], step):
        a, b = f[at:at + step].to(torch.complex128).conj(), x[at:at + step].to(torch.complex128)
        total += torch.stack([(a[:, i] * b[:, j]).sum() for i in range(2) for j in range(2)])
    return torch.view_as_real(total).reshape(-1)
