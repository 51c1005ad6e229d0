"""Performance cases: the work that users of the simulator have it do, through its public
entry points, over the range of sizes it serves.

`listed()` names the cases, `draw(rng)` gives one more of the same ranges, `prepare(case, seed)`
makes what a program holds before the call, `run(state)` is one pass through the entry points,
`work(case)` the bytes and operations the pass cannot do without, and `exact(case, seed)` the
same outputs from a plain torch complex128 simulation that uses none of the library's code.

Families (the "what" of a case):
  plan      a compiled circuit executed on a resident state (State.reset + State.execute)
  run       one request from the gate list to the answer (State.run, then the probabilities)
  batch     many small circuits of uneven size in persistent launches (Batch.run + read-out)
  gates     gate by gate through apply_1q / apply_controlled / apply_2q
  dense     fused k-qubit unitaries through apply_dense
  permute   PermuteQubits: a random reordering of all qubits, then a few local-global exchanges
Circuit constructions are those of the repository's workloads: RZ/RX layers with CZ pairs biased
toward high qubits, Haar 2x2 layers with CNOTs (or CNOT / CZ) on random matchings, random
H / Y / CNOT circuits of 30 n gates, and the textbook QFT.
"""
import math

import numpy as np
import torch

import paper_2010_09746_gb300 as qs


class Gate:
    """One gate as the binding takes it: kind, qubits, param, matrix."""
    __slots__ = ("kind", "qubits", "param", "matrix")

    def __init__(self, kind, qubits, param=0.0, matrix=None):
        self.kind, self.qubits, self.param, self.matrix = kind, qubits, param, matrix


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest compiled circuit: 12 qubits, 20 layers of Haar gates and CNOTs (one
        # shared-memory tile; latency and launches count)
        {"name": "plan_12q_haar_c128", "what": "plan", "circuit": "haar", "n": 12, "dtype": "c128", "layers": 20,
         "mode": "tile"},
        # a small served request, odd size: a handful of tiles on a 152-SM chip
        {"name": "plan_17q_mixed_c64", "what": "plan", "circuit": "mixed", "n": 17, "dtype": "c64", "layers": 60,
         "mode": "tile"},
        # an ordinary served request in double precision
        {"name": "plan_23q_mixed_c128", "what": "plan", "circuit": "mixed", "n": 23, "dtype": "c128", "layers": 50,
         "mode": "tile"},
        # the random-circuit workload in single precision, an ordinary large state
        {"name": "plan_27q_rzrx_c64", "what": "plan", "circuit": "rzrx", "n": 27, "dtype": "c64", "layers": 40,
         "mode": "tile"},
        # the headline workload: 30 qubits, double precision, 40 layers (16 GiB)
        {"name": "plan_30q_rzrx_c128", "what": "plan", "circuit": "rzrx", "n": 30, "dtype": "c128", "layers": 40,
         "mode": "tile"},
        # a structured algorithm: the textbook QFT (controlled phases and final SWAPs)
        {"name": "plan_25q_qft_c128", "what": "plan", "circuit": "qft", "n": 25, "dtype": "c128", "layers": 1,
         "mode": "tile"},
        # the paper's own compiler pass (Algorithm 1: permutations, tile passes, non-local gates)
        # on the paper's random circuits
        {"name": "paper_26q_random_c64", "what": "plan", "circuit": "random", "n": 26, "dtype": "c64", "layers": 1,
         "mode": "paper"},
        # one request from gate list to probabilities: compile, execute, read out
        {"name": "run_18q_mixed_c128", "what": "run", "circuit": "mixed", "n": 18, "dtype": "c128", "layers": 30},
        # many small circuits of uneven qubit count and depth
        {"name": "batch_192_c64", "what": "batch", "dtype": "c64", "count": 192, "nmin": 10, "nmax": 18, "dmin": 10,
         "dmax": 60},
        # gate by gate, double precision, 1 GiB state
        {"name": "gates_26q_c128", "what": "gates", "n": 26, "dtype": "c128"},
        # fused k-qubit unitaries, k = 2 .. 6, single precision, on low, middle and high qubits
        {"name": "dense_27q_c64", "what": "dense", "n": 27, "dtype": "c64", "kmax": 6},
        # qubit reordering of a 4 GiB state
        {"name": "permute_28q_c128", "what": "permute", "n": 28, "dtype": "c128"},
    ]


def draw(rng):
    what = rng.choice(["plan", "plan", "plan", "plan", "plan", "run", "batch", "gates", "gates", "dense", "dense",
                       "permute"])
    dtype = rng.choice(["c64", "c128"])
    if what == "plan":
        circuit = rng.choice(["haar", "mixed", "rzrx", "rzrx", "qft", "random"])
        mode = rng.choice(["tile", "paper"]) if circuit == "random" else "tile"
        n = rng.randint(12, {"haar": 22, "mixed": 25, "rzrx": 29, "qft": 28, "random": 27}[circuit])
        layers = {"haar": rng.randint(8, 24), "mixed": rng.randint(20, 60), "rzrx": rng.randint(10, 40)}.get(circuit, 1)
        return {"what": what, "circuit": circuit, "n": n, "dtype": dtype, "layers": layers, "mode": mode}
    if what == "run":
        return {"what": what, "circuit": rng.choice(["mixed", "rzrx", "haar"]), "n": rng.randint(10, 22), "dtype": dtype,
                "layers": rng.randint(5, 40)}
    if what == "batch":
        lo = rng.randint(10, 12)
        return {"what": what, "dtype": dtype, "count": rng.randint(40, 192), "nmin": lo, "nmax": lo + rng.randint(3, 6),
                "dmin": 10, "dmax": rng.randint(20, 60)}
    if what == "dense":
        return {"what": what, "n": rng.randint(12, 27), "dtype": dtype, "kmax": rng.randint(3, 6 if dtype == "c64" else 5)}
    return {"what": what, "n": rng.randint(10, 28), "dtype": dtype}


# ------------------------------------------------------------------------------------------
# circuits (gate lists, from the seed alone)
# ------------------------------------------------------------------------------------------
def _haar_2x2(count, rng):
    """count Haar-random 2x2 unitaries (Zyczkowski-Kus angles)."""
    f = np.arcsin(np.sqrt(rng.uniform(0.0, 1.0, count)))
    a, p, c = rng.uniform(0.0, 2.0 * math.pi, (3, count))
    m = np.empty((count, 2, 2), dtype=np.complex128)
    m[:, 0, 0] = np.exp(1j * (a + p)) * np.cos(f)
    m[:, 0, 1] = np.exp(1j * (a + c)) * np.sin(f)
    m[:, 1, 0] = -np.exp(1j * (a - c)) * np.sin(f)
    m[:, 1, 1] = np.exp(1j * (a - p)) * np.cos(f)
    return m


def _haar_unitary(dim, rng):
    z = (rng.standard_normal((dim, dim)) + 1j * rng.standard_normal((dim, dim))) / math.sqrt(2.0)
    q, r = np.linalg.qr(z)
    d = np.diag(r)
    return np.ascontiguousarray(q * (d / np.abs(d)))


def _circuit(name, n, layers, rng):
    out = []
    if name in ("haar", "mixed"):
        u = _haar_2x2(layers * n, rng)
        for k in range(layers):
            out += [Gate("U1", (q,), 0.0, u[k * n + q]) for q in range(n)]
            s = rng.permutation(n).tolist()
            cz = rng.uniform(size=n // 2) < 0.5
            out += [Gate("CZ" if name == "mixed" and cz[i] else "CNOT", (s[2 * i], s[2 * i + 1])) for i in range(n // 2)]
    elif name == "rzrx":
        w = (np.arange(n) + 1.0) ** 2
        t = rng.uniform(0.0, 2.0 * math.pi, (layers, n, 2))
        for k in range(layers):
            for q in range(n):
                out.append(Gate("RZ", (q,), float(t[k, q, 0])))
                out.append(Gate("RX", (q,), float(t[k, q, 1])))
            s = rng.choice(n, size=2 * (n // 4), replace=False, p=w / w.sum()).tolist()
            out += [Gate("CZ", (s[2 * i], s[2 * i + 1])) for i in range(n // 4)]
    elif name == "random":
        for _ in range(30 * n):
            if rng.uniform() < 0.3:
                a, b = rng.choice(n, size=2, replace=False).tolist()
                out.append(Gate("CNOT", (a, b)))
            else:
                out.append(Gate("H" if rng.uniform() < 0.5 else "Y", (int(rng.integers(n)),)))
    elif name == "qft":
        # a product state to transform, then the QFT
        out += [Gate("U1", (q,), 0.0, m) for q, m in enumerate(_haar_2x2(n, rng))]
        for j in range(n - 1, -1, -1):
            out.append(Gate("H", (j,)))
            out += [Gate("CP", (k, j), math.pi / (1 << (j - k))) for k in range(j - 1, -1, -1)]
        out += [Gate("SWAP", (j, n - 1 - j)) for j in range(n // 2)]
    else:
        raise ValueError(name)
    return out


def _batch_circuits(case, seed):
    rng = np.random.default_rng([seed, 2])
    # the sizes belong to the case (every state of it costs the same), the gates to the seed
    shape = np.random.default_rng([case["count"], case["nmin"], case["nmax"], case["dmin"], case["dmax"]])
    ns = shape.integers(case["nmin"], case["nmax"] + 1, case["count"]).tolist()
    ds = shape.integers(case["dmin"], case["dmax"] + 1, case["count"]).tolist()
    return [(n, _circuit("mixed", n, d, rng)) for n, d in zip(ns, ds)]


def _gate_calls(n, rng):
    """1-qubit, controlled and 2-qubit gates on low, middle and high qubits."""
    u = _haar_2x2(7, rng)
    lo, mid, hi = 1, n // 2, n - 1
    return ([("1q", u[0], (0,)), ("1q", u[1], (mid,)), ("1q", u[2], (hi,)), ("1q", u[3], (lo + 1,)),
             ("c", u[4], (mid, lo)), ("c", u[5], (0, hi)), ("c", u[6], (hi - 1, mid + 1))]
            + [("2q", _haar_unitary(4, rng), q) for q in ((0, 1), (lo, hi), (hi, mid))])


def _dense_calls(n, kmax, rng):
    """k-qubit unitaries, each k on low qubits and on qubits spread over the register."""
    out = []
    for k in range(2, kmax + 1):
        spread = [(n - 1) * i // (k - 1) for i in range(k)][::-1]
        out.append((_haar_unitary(1 << k, rng), list(range(k))))
        out.append((_haar_unitary(1 << k, rng), spread))
    return out


def _permutations(n, rng):
    p = rng.permutation(n).tolist()
    q = list(p)
    for k in range(min(3, n // 4)):   # exchange a few low storage bits with high ones
        a, b = q.index(k), q.index(n - 1 - k)
        q[a], q[b] = q[b], q[a]
    return p, q


def _random_state(n, seed, device="cuda"):
    """A normalised complex Gaussian vector, float64 pairs, made on the device."""
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    v = torch.randn((1 << n, 2), generator=g, device=device, dtype=torch.float64)
    v *= 1.0 / float(torch.linalg.vector_norm(v))
    return v


# ------------------------------------------------------------------------------------------
# states and passes
# ------------------------------------------------------------------------------------------
class _Amplitudes:
    """A state's amplitude vector for torch.as_tensor: (re, im) rows.  torch keeps this object, and
    with it the state that owns the memory, for as long as the tensor lives."""

    def __init__(self, st):
        self.state = st
        self.__cuda_array_interface__ = {"data": (st.device_ptr(), False), "shape": (1 << st.n, 2),
                                         "typestr": "<f8" if st.dtype == qs.QS_C128 else "<f4", "version": 3}


def _view(st):
    """The state's amplitude vector as a torch tensor of (re, im) rows, no copy."""
    return torch.as_tensor(_Amplitudes(st), device="cuda")


def prepare(case, seed):
    what = case["what"]
    rng = np.random.default_rng([seed, 1])
    s = {"what": what}
    if what == "batch":
        s["batch"] = qs.Batch(_batch_circuits(case, seed), dtype=case["dtype"])
        return s
    n = case["n"]
    s["state"] = st = qs.State(n, case["dtype"])
    s["identity"] = list(range(n))
    if what == "plan":
        s["plan"] = qs.compile(n, _circuit(case["circuit"], n, case["layers"], rng), mode=case["mode"],
                               dtype=case["dtype"])
    elif what == "run":
        s["circuit"] = _circuit(case["circuit"], n, case["layers"], rng)
    else:
        v = _view(st)
        v.copy_(_random_state(n, seed))
        torch.cuda.synchronize()
        if what == "gates":
            s["calls"] = _gate_calls(n, rng)
        elif what == "dense":
            s["calls"] = _dense_calls(n, case["kmax"], rng)
        else:
            s["perms"] = _permutations(n, rng)
    return s


def run(s):
    what = s["what"]
    if what == "batch":
        b = s["batch"]
        b.run()
        return {"norms": b.norms(), "amplitudes": np.concatenate([b.amplitudes(i) for i in range(b.count)])}
    st = s["state"]
    if what == "plan":
        st.reset()
        st.execute(s["plan"])
        st.permute(s["identity"])   # logical order (nothing to move unless the plan permuted)
    elif what == "run":
        st.reset()
        st.run(s["circuit"])
        return {"probabilities": st.probabilities(), "norm": st.norm()}
    elif what == "gates":
        for kind, u, q in s["calls"]:
            if kind == "1q":
                st.apply_1q(u, q[0])
            elif kind == "c":
                st.apply_controlled(u, q[0], q[1])
            else:
                st.apply_2q(u, q[0], q[1])
    elif what == "dense":
        for u, q in s["calls"]:
            st.apply_dense(u, q)
        st.permute(s["identity"])
    else:
        for p in s["perms"]:
            st.permute(p)
    return _view(st)


# ------------------------------------------------------------------------------------------
# the work of a pass
# ------------------------------------------------------------------------------------------
def _gate_flops(g):
    """Real operations per amplitude of one gate as the method writes it."""
    if g.kind in ("CNOT", "CZ", "SWAP", "Y", "X"):
        return 0.0
    if g.kind == "RZ":
        return 6.0
    if g.kind == "CP":
        return 1.5
    return 14.0


def work(case):
    what = case["what"]
    elem = 16 if case["dtype"] == "c128" else 8
    if what == "batch":
        cs = _batch_circuits(case, 0)
        return {"bytes": float(sum(elem << n for n, _ in cs)),
                "flops": sum(sum(map(_gate_flops, c)) * (1 << n) for n, c in cs)}
    n = case["n"]
    N = 1 << n
    if what in ("plan", "run"):   # |0...0> is not read; the final state (or its probabilities) is written
        fl = sum(map(_gate_flops, _circuit(case["circuit"], n, case["layers"], np.random.default_rng(0)))) * N
        return {"bytes": float(N * (8 if what == "run" else elem)), "flops": fl}
    if what == "gates":   # each call reads and writes what it changes (a controlled gate half of the state)
        return {"bytes": (4 + 3 * 0.5 + 3) * 2.0 * N * elem, "flops": (4 * 14 + 3 * 7 + 3 * 30) * float(N)}
    if what == "dense":
        ks = range(2, case["kmax"] + 1)
        return {"bytes": 2.0 * len(ks) * 2.0 * N * elem, "flops": sum(2 * (8.0 * (1 << k) - 2) for k in ks) * N}
    return {"bytes": 2 * 2.0 * N * elem, "flops": 0.0}


# ------------------------------------------------------------------------------------------
# the same outputs in 64 bits, plain torch
# ------------------------------------------------------------------------------------------
_S = 1.0 / math.sqrt(2.0)
_NAMED = {"H": np.array([[_S, _S], [_S, -_S]], dtype=np.complex128), "Y": np.array([[0, -1j], [1j, 0]])}


def _matrix_1q(g):
    if g.matrix is not None:
        return g.matrix
    t = 0.5 * g.param
    if g.kind == "RZ":
        return np.diag([np.exp(-1j * t), np.exp(1j * t)])
    if g.kind == "RX":
        return np.array([[math.cos(t), -1j * math.sin(t)], [-1j * math.sin(t), math.cos(t)]])
    return _NAMED[g.kind]


def _axes(psi, n, qubits):
    """The vector as an n-axis tensor's view with the qubits' axes first (first listed qubit last
    among them: least significant), the others grouped."""
    qs_sorted = sorted(qubits, reverse=True)
    shape, prev = [], n
    for q in qs_sorted:
        shape += [1 << (prev - 1 - q), 2]
        prev = q
    shape.append(1 << prev)
    v = psi.view(shape)
    pos = {q: 2 * i + 1 for i, q in enumerate(qs_sorted)}
    rest = [i for i in range(len(shape)) if i not in pos.values()]
    return v.permute([pos[q] for q in reversed(list(qubits))] + rest)


def _apply(psi, n, u, qubits):
    """The 2^k x 2^k matrix u on the listed qubits (first = least significant), in place."""
    k = len(qubits)
    v = _axes(psi, n, qubits)
    D = 1 << k
    idx = [tuple((r >> (k - 1 - i)) & 1 for i in range(k)) for r in range(D)]
    if k <= 2:
        x = [v[i].clone() for i in idx]
        for r in range(D):
            acc = x[0] * complex(u[r, 0])
            for c in range(1, D):
                if u[r, c] != 0:
                    acc.add_(x[c], alpha=complex(u[r, c]))
            v[idx[r]] = acc
        return
    m = torch.as_tensor(np.ascontiguousarray(u), device=psi.device)
    y = m @ v.reshape(D, -1)
    v.copy_(y.view(v.shape))


def _simulate(n, circuit, device="cuda"):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device=device)
    psi[0] = 1.0
    pend = {}

    def flush(q):
        u = pend.pop(q, None)
        if u is not None:
            _apply(psi, n, u, (q,))

    for g in circuit:
        if len(g.qubits) == 1:
            q = g.qubits[0]
            pend[q] = _matrix_1q(g) @ pend[q] if q in pend else _matrix_1q(g)
            continue
        for q in g.qubits:
            flush(q)
        v = _axes(psi, n, (g.qubits[1], g.qubits[0]))   # axes: (first listed, second listed, rest)
        if g.kind == "CZ":
            v[1, 1] *= -1
        elif g.kind == "CP":
            v[1, 1] *= complex(math.cos(g.param), math.sin(g.param))
        elif g.kind == "CNOT":
            t = v[1, 0].clone()
            v[1, 0] = v[1, 1]
            v[1, 1] = t
        else:   # SWAP
            t = v[0, 1].clone()
            v[0, 1] = v[1, 0]
            v[1, 0] = t
    for q in list(pend):
        flush(q)
    return psi


def _logical_to_storage(psi, n, perm):
    """Amplitude i at component sum_q i_q 2^perm[q]."""
    v = psi.view([2] * n)   # axis a holds qubit n - 1 - a
    inv = [0] * n
    for q, p in enumerate(perm):
        inv[p] = q
    return v.permute([n - 1 - inv[n - 1 - a] for a in range(n)]).reshape(-1)


def exact(case, seed):
    what = case["what"]
    rng = np.random.default_rng([seed, 1])
    if what == "batch":
        psis = [_simulate(n, c) for n, c in _batch_circuits(case, seed)]
        return {"norms": np.array([float(torch.linalg.vector_norm(p)) ** 2 for p in psis]),
                "amplitudes": np.concatenate([p.cpu().numpy() for p in psis])}
    n = case["n"]
    if what in ("plan", "run"):
        c = _circuit(case["circuit"], n, case["layers"], rng)
        if len(c) * (96.0 * (1 << n)) / 3e12 > 15.0:   # about the seconds it takes
            return None
        psi = _simulate(n, c)
        if what == "run":
            p = torch.view_as_real(psi).square().sum(1)
            return {"probabilities": p.cpu().numpy(), "norm": float(p.sum())}
        return torch.view_as_real(psi)
    psi = torch.view_as_complex(_random_state(n, seed).to(torch.float32 if case["dtype"] == "c64" else torch.float64)
                                .to(torch.float64))
    if what == "gates":
        for kind, u, q in _gate_calls(n, rng):
            if kind == "c":
                v = _axes(psi, n, (q[1], q[0]))[1]
                a, b = v[0].clone(), v[1].clone()
                v[0] = a * complex(u[0, 0]) + b * complex(u[0, 1])
                v[1] = a * complex(u[1, 0]) + b * complex(u[1, 1])
            else:
                _apply(psi, n, u, q)
    elif what == "dense":
        for u, q in _dense_calls(n, case["kmax"], rng):
            _apply(psi, n, u, q)
    else:
        psi = _logical_to_storage(psi, n, _permutations(n, rng)[1])
    return torch.view_as_real(psi)
