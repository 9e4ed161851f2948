"""The workloads whose speed this framework is judged by, each through its public entry points.

A case is a dict of plain values.  Its `kind` says which use it stands for:

* ``circuit``  -- set a basis state, apply a fused (or unfused) circuit, leave the state in
  the caller's buffer; families brickwork, grid, qft, qft_brickwork (the circuits of the
  tests and of the benchmark, drawn here from their own seeds);
* ``noise``    -- the same with a density matrix: a noisy grid circuit on n qubits as a
  2n-qubit vector, and its outcome distribution;
* ``batch``    -- a parameter sweep: many hardware-efficient circuits of one shape, each with
  its own angles, and the energy of each;
* ``energy``   -- the expectation value of a transverse-field Ising chain (n - 1 ZZ terms and
  n X terms), the inner call of a variational loop;
* ``readout``  -- what is read from a finished state: norm, probabilities, the most probable
  outcomes, shots.

Circuits are fused when the state is prepared: a program keeps the schedule and applies it
many times.  The seed draws the angles, the gate choice, the basis state and the amplitudes.
"""
import math

import numpy as np
import torch

C64, C128 = "c64", "c128"

# Register widths from a few qubits, where a call is latency and launches, over the tests'
# and the benchmark's 12, 16-22 and 24 qubits, up to the 28 qubits where its headline range
# begins (2 GiB of complex64, 4 GiB of complex128 per state).
_LISTED = [
    # the 12-qubit brickwork circuit, complex128, gate by gate: the reference form of every
    # small study (350 gates on a 64 KiB state)
    {"name": "brickwork_12q_c128_unfused", "kind": "circuit", "family": "brickwork", "n": 12, "layers": 20,
     "k": 0, "dtype": C128},
    # the same circuit as a user runs it for speed: complex64, fused to width 5
    {"name": "brickwork_12q_c64_k5", "kind": "circuit", "family": "brickwork", "n": 12, "layers": 20, "k": 5,
     "dtype": C64},
    # an ordinary mid-size run, state smaller than L2: 20 qubits of the grid circuit, complex64
    {"name": "grid_20q_c64_k5", "kind": "circuit", "family": "grid", "n": 20, "layers": 24, "k": 5, "dtype": C64},
    # mid-size in complex128, diagonal, permutation and dense gates mixed: QFT and U3 / CNOT
    # ladder layers on an odd width
    {"name": "qft_brickwork_23q_c128_k4", "kind": "circuit", "family": "qft_brickwork", "n": 23, "layers": 4, "k": 4,
     "dtype": C128},
    # the headline workload at the lower end of its range: 28 qubits, depth 24, width 5,
    # complex64 with the norm-drift check
    {"name": "grid_28q_c64_k5", "kind": "circuit", "family": "grid", "n": 28, "layers": 24, "k": 5, "dtype": C64,
     "adaptive": True},
    # the same in complex128, fused to width 4
    {"name": "grid_28q_c128_k4", "kind": "circuit", "family": "grid", "n": 28, "layers": 24, "k": 4, "dtype": C128},
    # a large QFT: almost all gates are controlled phases
    {"name": "qft_28q_c64_k5", "kind": "circuit", "family": "qft", "n": 28, "layers": 0, "k": 5, "dtype": C64},
    # a noisy grid circuit on 12 qubits: the density matrix is a 24-qubit vector
    {"name": "noise_12q_c64_k5", "kind": "noise", "n": 12, "layers": 8, "k": 5, "p": 0.01, "dtype": C64},
    # a parameter sweep: 96 circuits of 18 qubits and their energies
    {"name": "batch_18q_x96_c64_k5", "kind": "batch", "n": 18, "count": 96, "layers": 6, "k": 5, "dtype": C64},
    # the energy of a 26-qubit chain
    {"name": "energy_26q_c64", "kind": "energy", "n": 26, "dtype": C64},
    # reading out a large state, and a small one, where every call is latency
    {"name": "readout_28q_c64", "kind": "readout", "n": 28, "topk": 64, "shots": 1 << 20, "dtype": C64},
    {"name": "readout_13q_c64", "kind": "readout", "n": 13, "topk": 64, "shots": 1000, "dtype": C64},
]


def listed():
    return [dict(c) for c in _LISTED]


def draw(rng):
    """One more case of the listed ones' ranges."""
    kind = rng.choice(["brickwork", "grid", "grid", "qft_brickwork", "qft", "noise", "batch", "energy", "readout"])
    dtype = rng.choice([C64, C64, C128])
    top = 28 if dtype == C64 else 27          # widest register: the same bytes
    if kind == "brickwork":
        return {"kind": "circuit", "family": kind, "n": rng.randint(3, 17), "layers": rng.randint(3, 24),
                "k": rng.randint(0, 5), "dtype": dtype}
    if kind == "grid":
        return {"kind": "circuit", "family": kind, "n": rng.randint(13, top), "layers": rng.randint(4, 24),
                "k": rng.randint(3, 5), "dtype": dtype, "adaptive": rng.random() < 0.3}
    if kind == "qft_brickwork":
        return {"kind": "circuit", "family": kind, "n": rng.randint(8, top - 3), "layers": rng.randint(1, 8),
                "k": rng.randint(2, 5), "dtype": dtype}
    if kind == "qft":
        return {"kind": "circuit", "family": kind, "n": rng.randint(9, top), "layers": 0, "k": rng.randint(2, 5),
                "dtype": dtype}
    if kind == "noise":
        return {"kind": "noise", "n": rng.randint(3, 13), "layers": rng.randint(2, 8), "k": rng.randint(3, 5),
                "p": 10.0 ** rng.uniform(-4, -1), "dtype": dtype}
    if kind == "batch":
        n = rng.randint(8, 21)
        most = max(2, min(200, 1 << (25 - n)))
        return {"kind": "batch", "n": n, "count": max(2, int(most ** rng.uniform(0.3, 1.0))), "layers": rng.randint(2, 6),
                "k": rng.choice([3, 4, 5, 5]), "dtype": dtype}
    if kind == "energy":
        return {"kind": "energy", "n": rng.randint(3, top - 1), "dtype": dtype}
    return {"kind": "readout", "n": rng.randint(3, top), "topk": rng.randint(1, 64),
            "shots": int(2 ** rng.uniform(0, 20)), "dtype": dtype}


# ------------------------------------------------------------------ circuits, in plain numpy
# A gate is (qubits, matrix): local bit j of the matrix is qubits[j], qubit t is bit t of the
# amplitude's index.

_H = np.array([[1, 1], [1, -1]], dtype=np.complex128) / math.sqrt(2.0)
_X = np.array([[0, 1], [1, 0]], dtype=np.complex128)
_Y = np.array([[0, -1j], [1j, 0]], dtype=np.complex128)
_Z = np.diag([1.0, -1.0]).astype(np.complex128)
_ROOTS = [((1 + 1j) * np.eye(2) + (1 - 1j) * p) / 2 for p in (_X, _Y, (_X + _Y) / math.sqrt(2.0))]
_CNOT = np.eye(4, dtype=np.complex128)[[0, 3, 2, 1]]           # control: local bit 0
_SWAP = np.eye(4, dtype=np.complex128)[[0, 2, 1, 3]]
_CZ = np.diag([1.0, 1.0, 1.0, -1.0]).astype(np.complex128)


def _cp(phi):
    return np.diag([1.0, 1.0, 1.0, complex(math.cos(phi), math.sin(phi))]).astype(np.complex128)


def _u3(t, p, q):
    c, s = math.cos(t / 2), math.sin(t / 2)
    return np.array([[c, -np.exp(1j * q) * s], [np.exp(1j * p) * s, np.exp(1j * (p + q)) * c]], dtype=np.complex128)


def _fsim(t, p):
    m = np.zeros((4, 4), dtype=np.complex128)
    m[0, 0], m[3, 3] = 1.0, np.exp(-1j * p)
    m[1, 1] = m[2, 2] = math.cos(t)
    m[1, 2] = m[2, 1] = -1j * math.sin(t)
    return m


def _qft(n):
    gates = []
    for j in range(n - 1, -1, -1):
        gates.append(((j,), _H))
        gates += [((k, j), _cp(math.pi / 2 ** (j - k))) for k in range(j - 1, -1, -1)]
    return gates + [((i, n - 1 - i), _SWAP) for i in range(n // 2)]


def _grid(n, cycles, rng):
    cols = int(math.ceil(math.sqrt(n)))
    gates, f = [], _fsim(math.pi / 2, math.pi / 6)
    for cyc in range(cycles):
        gates += [((q,), _ROOTS[int(c)]) for q, c in enumerate(rng.integers(0, 3, size=n))]
        for q in range(n):
            r, c = divmod(q, cols)
            a = cyc % 4
            if a < 2 and c + 1 < cols and q + 1 < n and c % 2 == a:
                gates.append(((q, q + 1), f))
            if a >= 2 and q + cols < n and r % 2 == a - 2:
                gates.append(((q, q + cols), f))
    return gates


def _u3_layers(n, layers, rng, pairs, two):
    gates = []
    for layer in range(layers):
        ang = rng.uniform(0.0, 2.0 * math.pi, size=(n, 3))
        gates += [((q,), _u3(*ang[q])) for q in range(n)]
        gates += [((i, i + 1), two) for i in pairs(layer)]
    return gates


def _circuit(case, rng):
    n, layers = case["n"], case["layers"]
    if case["family"] == "brickwork":
        return _u3_layers(n, layers, rng, lambda layer: range(layer % 2, n - 1, 2), _CZ)
    if case["family"] == "grid":
        return _grid(n, layers, rng)
    gates = _qft(n)
    return gates + _u3_layers(n, layers, rng, lambda layer: range(n - 1), _CNOT) if layers else gates


def _hea(n, layers, rng):
    gates = []
    for _ in range(layers):
        t, p = rng.uniform(-math.pi, math.pi, size=n), rng.uniform(-math.pi, math.pi, size=n)
        for q in range(n):
            c, s = math.cos(t[q] / 2), math.sin(t[q] / 2)
            gates.append(((q,), np.array([[c, -s], [s, c]], dtype=np.complex128)))
            gates.append(((q,), np.diag([np.exp(-0.5j * p[q]), np.exp(0.5j * p[q])])))
        gates += [((i, i + 1), _CNOT) for i in range(n - 1)]
    return gates


def _rng(case, seed):
    return np.random.default_rng([int(seed) & 0xFFFFFFFF, case["n"]])


def _zz(n):
    """The open chain sum_i Z_i Z_{i+1} as X masks, Z masks and coefficients."""
    return [0] * (n - 1), [3 << i for i in range(n - 1)], [1.0] * (n - 1)


def _ising(n, rng):
    """-sum J_i Z_i Z_{i+1} - sum h_i X_i with seeded couplings near 1."""
    j, h = rng.uniform(0.8, 1.2, size=n - 1), rng.uniform(0.5, 1.5, size=n)
    return ([0] * (n - 1) + [1 << i for i in range(n)], [3 << i for i in range(n - 1)] + [0] * n,
            [-float(v) for v in j] + [-float(v) for v in h])


def _real(dtype):
    return torch.float32 if dtype == C64 else torch.float64


def _complex(dtype):
    return torch.complex64 if dtype == C64 else torch.complex128


def _random_state(case, seed):
    """A random state: complex normal amplitudes, norm 1."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    v = torch.randn((1 << case["n"], 2), generator=g, device="cuda", dtype=_real(case["dtype"]))
    v /= float(torch.linalg.vector_norm(v, dtype=torch.float64))
    return torch.view_as_complex(v)


def _ansatz_state(case, seed):
    """A variational state: a product of seeded rotations with 30% of noise on every amplitude."""
    rng, n = _rng(case, seed), case["n"]
    t, p = rng.uniform(0.2, 1.1, size=n), rng.uniform(-0.5, 0.5, size=n)
    v = torch.ones(1, device="cuda", dtype=torch.complex128)
    for q in range(n):
        pair = torch.tensor([math.cos(t[q] / 2), math.sin(t[q] / 2) * complex(math.cos(p[q]), math.sin(p[q]))],
                            device="cuda", dtype=torch.complex128)
        v = (pair[:, None] * v[None, :]).reshape(-1)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    v = v.to(_complex(case["dtype"]))
    noise = torch.view_as_complex(torch.randn((1 << n, 2), generator=g, device="cuda", dtype=_real(case["dtype"])))
    v = v * (1.0 + 0.3 * noise)
    return v / float(torch.linalg.vector_norm(torch.view_as_real(v), dtype=torch.float64))


# ------------------------------------------------------------------ prepare, run, work

def prepare(case, seed):
    from paper_2604_03816_gb300 import sv

    n, kind, stream = case["n"], case["kind"], torch.cuda.current_stream()
    dt = sv.SV_C64 if case["dtype"] == C64 else sv.SV_C128
    rng = _rng(case, seed)
    s = {"sv": sv, "case": case, "x": int(rng.integers(0, 1 << n))}
    if kind == "circuit":
        s["out"] = torch.empty(1 << n, device="cuda", dtype=_complex(case["dtype"]))
        s["circuit"] = sv.sv_fuse(_circuit(case, rng), n, case["k"])
        s["state"] = sv.sv_alloc(n, dt, dev_buf=s["out"], stream=stream)
    elif kind == "noise":
        s["rho"] = torch.empty(1 << (2 * n), device="cuda", dtype=_complex(case["dtype"]))
        s["p"] = torch.empty(1 << n, device="cuda", dtype=_real(case["dtype"]))
        s["circuit"] = sv.sv_fuse_density(_grid(n, case["layers"], rng), n, case["p"], case["k"])
        s["state"] = sv.sv_alloc(2 * n, dt, dev_buf=s["rho"], stream=stream)
    elif kind == "batch":
        s["out"] = torch.empty((case["count"], 1 << n), device="cuda", dtype=_complex(case["dtype"]))
        first = sv.sv_fuse(_hea(n, case["layers"], rng), n, case["k"])
        s["circuits"] = [first] + [sv.sv_fuse_like(first, _hea(n, case["layers"], rng)) for _ in range(case["count"] - 1)]
        s["batch"] = sv.sv_batch_alloc(n, dt, case["count"], dev_buf=s["out"], stream=stream)
    else:
        s["psi"] = _ansatz_state(case, seed) if kind == "energy" else _random_state(case, seed)
        s["state"] = sv.sv_alloc(n, dt, stream=stream)
        sv.sv_set_state(s["state"], s["psi"])
        sv.sv_sync(s["state"])
        s["psi"] = None
        if kind == "energy":
            s["terms"] = _ising(n, rng)
        else:
            s["probs"] = torch.empty(1 << n, device="cuda", dtype=_real(case["dtype"]))
            s["shots"] = torch.empty(case["shots"], device="cuda", dtype=torch.int64)
            s["seed"] = int(seed)
    return s


def run(state):
    sv, case = state["sv"], state["case"]
    kind = case["kind"]
    if kind == "circuit":
        sv.sv_set_basis(state["state"], state["x"])
        sv.sv_apply_circuit(state["state"], state["circuit"], adaptive=bool(case.get("adaptive", False)))
        return state["out"]
    if kind == "noise":
        sv.sv_set_basis(state["state"], 0)
        sv.sv_apply_circuit(state["state"], state["circuit"])
        return {"rho": state["rho"], "p": sv.sv_density_probs(state["state"], out=state["p"])}
    if kind == "batch":
        sv.sv_batch_set_basis(state["batch"], 0)
        # 512 MiB chunks: what the autotuner picks for these widths
        sv.sv_batch_apply(state["batch"], state["circuits"], l2_bytes=1 << 29)
        energy = sv.sv_batch_expect(state["batch"], *_zz(case["n"]))
        # complex64 amplitudes carry no more digits than FP32 into an energy
        return {"psi": state["out"], "energy": energy.astype(np.float32) if case["dtype"] == C64 else energy}
    if kind == "energy":
        return sv.sv_expect(state["state"], *state["terms"])
    idx, p = sv.sv_topk(state["state"], case["topk"])
    return {"norm": sv.sv_norm(state["state"]), "idx": idx.astype(np.int64), "p": p,
            "probs": sv.sv_probs(state["state"], out=state["probs"]),
            "shots": sv.sv_sample(state["state"], state["seed"], case["shots"], out=state["shots"])}


def work(case):
    """Bytes: the state (or the batch) read or written once, the results written once.
    Operations: the gates of the circuit as given (unfused), 8 2^k per amplitude for a gate on
    k qubits, 6 per amplitude that a diagonal gate changes."""
    n, kind, amp = case["n"], case["kind"], 8 if case["dtype"] == C64 else 16
    rng = np.random.default_rng(0)

    def flops(gates):
        f = 0.0
        for q, u in gates:
            d = np.diag(u)
            diagonal = np.count_nonzero(u) == np.count_nonzero(d) == len(d)
            f += 6.0 * float(np.mean(d != 1)) if diagonal else 8.0 * len(d)
        return f

    if kind == "circuit":
        return {"bytes": amp << n, "flops": flops(_circuit(case, rng)) * 2.0 ** n}
    if kind == "noise":
        gates = _grid(n, case["layers"], rng)
        each = sum(2 * 8.0 * 2 ** len(q) + 4.0 * len(q) * 8 for q, _ in gates)
        return {"bytes": (amp << (2 * n)) + (amp // 2 << n), "flops": each * 4.0 ** n}
    if kind == "batch":
        return {"bytes": case["count"] * ((amp << n) + 8),
                "flops": case["count"] * (flops(_hea(n, case["layers"], rng)) + n + 2) * 2.0 ** n}
    if kind == "energy":
        return {"bytes": amp << n, "flops": (3 + (n - 1) + 4 * n) * 2.0 ** n}
    return {"bytes": (amp << n) + (amp // 2 << n) + 8 * case["shots"], "flops": 4.0 * 2 ** n}


# ------------------------------------------------------------------ the same in 64 bits

def _apply(v, n, qubits, u):
    """U on `qubits` (one or two) of the vector v, in place, plain torch."""
    d = np.diag(u)
    k = len(qubits)
    order = sorted(range(k), key=lambda j: -qubits[j])          # axes from the highest qubit
    shape, last = [], n
    for j in order:
        shape += [1 << (last - 1 - qubits[j]), 2]
        last = qubits[j]
    t = v.view(shape + [1 << last])

    def part(l):
        at = [slice(None)] * t.dim()
        for i, j in enumerate(order):
            at[2 * i + 1] = (l >> j) & 1
        return t[tuple(at)]

    if np.count_nonzero(u) == np.count_nonzero(d):
        for l in range(1 << k):
            if d[l] != 1:
                part(l).mul_(complex(d[l]))
        return
    old = [part(l).clone() for l in range(1 << k)]
    for r in range(1 << k):
        to = part(r)
        if u[r, r] != 0:
            to.mul_(complex(u[r, r]))
        else:
            to.zero_()
        for c in range(1 << k):
            if c != r and u[r, c] != 0:
                to.add_(old[c], alpha=complex(u[r, c]))


def _simulate(n, gates, x):
    """The circuit on |x>; one-qubit gates wait for the next two-qubit gate on their qubit."""
    v = torch.zeros(1 << n, device="cuda", dtype=torch.complex128)
    v[x] = 1.0
    wait = {}
    for q, u in gates:
        if len(q) == 1:
            wait[q[0]] = u @ wait.get(q[0], np.eye(2))
            continue
        a, b = wait.pop(q[0], None), wait.pop(q[1], None)
        if a is not None or b is not None:
            u = u @ np.kron(np.eye(2) if b is None else b, np.eye(2) if a is None else a)
        _apply(v, n, q, u)
    for q, u in wait.items():
        _apply(v, n, (q,), u)
    return v



def _zz_of(p, n, i):
    """sum_k (-1)^(k_i + k_(i+1)) p_k."""
    t = p.view(1 << (n - 2 - i), 4, 1 << i).sum(dim=2).sum(dim=0)
    return float(t[0] - t[1] - t[2] + t[3])


def exact(case, seed):
    n, kind = case["n"], case["kind"]
    rng = _rng(case, seed)
    x = int(rng.integers(0, 1 << n))
    if kind == "circuit":
        return _simulate(n, _circuit(case, rng), x)
    if kind == "noise":
        p = case["p"]
        channel = (1 - p) * np.eye(4, dtype=np.complex128) + (p / 3) * sum(np.kron(m.conj(), m) for m in (_X, _Y, _Z))
        gates = []
        for q, u in _grid(n, case["layers"], rng):
            gates += [(q, u), (tuple(t + n for t in q), u.conj())] + [((t, t + n), channel) for t in q]
        rho = _simulate(2 * n, gates, 0)
        return {"rho": rho, "p": rho.view(1 << n, 1 << n).diagonal().real.contiguous()}
    if kind == "batch":
        psi = torch.stack([_simulate(n, _hea(n, case["layers"], rng), 0) for _ in range(case["count"])])
        p = psi.real ** 2 + psi.imag ** 2
        return {"psi": psi, "energy": np.array([sum(_zz_of(r, n, i) for i in range(n - 1)) for r in p])}
    v = (_ansatz_state(case, seed) if kind == "energy" else _random_state(case, seed)).to(torch.complex128)
    p = v.real ** 2 + v.imag ** 2
    if kind == "energy":
        _, _, coef = _ising(n, rng)
        e = sum(c * _zz_of(p, n, i) for i, c in enumerate(coef[:n - 1]))
        for i, c in enumerate(coef[n - 1:]):
            t = v.view(-1, 2, 1 << i)
            e += c * 2.0 * float((t[:, 0].real * t[:, 1].real + t[:, 0].imag * t[:, 1].imag).sum())
        return e
    top = torch.topk(p, min(case["topk"], 1 << n)).values.cpu().numpy()
    return {"norm": float(p.sum()), "idx": None, "p": top, "probs": p, "shots": None}
