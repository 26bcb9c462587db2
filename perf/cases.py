"""The work that users have this simulator do, as timed cases.

A case is a dict of plain values; its ``kind`` names the use:

* ``gates``    a circuit applied gate by gate from |0...0>, then the parity probabilities of all qubits
               (the plain way to run a circuit; at 16 qubits every call is a launch, at 28 a pass over 2 GiB);
* ``dense``    dense gates on random target sets of one width, applied to a random state;
* ``fused``    a circuit in one fused call from |0...0>, in the state's own precision or on the tensor cores;
* ``energy``   one Trotter step of a few Pauli rotations, then the expectation value of every term;
* ``measure``  <Z_q> of every qubit, samples, then a parity measurement that collapses the state;
* ``batch``    many independent variational circuits and their observables in one launch.

Circuits, target sets, angles and states are drawn from the seed alone. Values that belong to a complex64 state
(probabilities, expectation values) are kept in single precision, as a program that chose that state type keeps
them; those of a complex128 state stay in double precision.
"""
import math

import numpy as np
import torch

from paper_2308_01999_gb300 import inputs as gen
from paper_2308_01999_gb300 import sv

PREC = {"native": sv.SV_PREC_NATIVE, "tf32": sv.SV_PREC_TF32, "split_bf16": sv.SV_PREC_SPLIT_BF16}


def listed():
    return [
        # the smallest calls: a 16-qubit circuit of 300 gates, one call and one launch each, and its parity
        {"name": "gates16", "kind": "gates", "dtype": "complex64", "n": 16, "gates": 300, "two": "cz,cnot"},
        # an ordinary large circuit, gate by gate: two layers (84 gates) on a 2 GiB state
        {"name": "gates28", "kind": "gates", "dtype": "complex64", "n": 28, "gates": 84, "two": "cz,cnot,crz"},
        # the same in double precision, the reference runs of a study: 1 GiB, 78 gates
        {"name": "gates26_c128", "kind": "gates", "dtype": "complex128", "n": 26, "gates": 78, "two": "cz,cnot,crz"},
        # wide dense gates on random targets, as the gate-application experiment applies them
        {"name": "dense5_28", "kind": "dense", "dtype": "complex64", "n": 28, "k": 5, "sets": 3},
        # a medium request of the serving path: 20 qubits, depth 24, one fused call at width 4
        {"name": "fused4_20", "kind": "fused", "dtype": "complex64", "n": 20, "form": "layered", "layers": 24, "w": 4,
         "prec": "native"},
        # fused brick wall at full width in the state's own precision
        {"name": "fused6_27", "kind": "fused", "dtype": "complex64", "n": 27, "form": "brick", "layers": 6, "w": 6,
         "prec": "native"},
        # the same at the two tensor-core precisions
        {"name": "fused6_28_tf32", "kind": "fused", "dtype": "complex64", "n": 28, "form": "brick", "layers": 8, "w": 6,
         "prec": "tf32"},
        {"name": "fused5_25_bf16", "kind": "fused", "dtype": "complex64", "n": 25, "form": "brick", "layers": 10, "w": 5,
         "prec": "split_bf16"},
        # a fused circuit in double precision
        {"name": "fused4_24_c128", "kind": "fused", "dtype": "complex128", "n": 24, "form": "layered", "layers": 5, "w": 4,
         "prec": "native"},
        # time evolution under a fermionic Hamiltonian: rotations, then the energy's terms
        {"name": "energy28", "kind": "energy", "dtype": "complex64", "n": 28, "form": "hopping", "rotations": 6,
         "strings": 24},
        # what is read off a random-circuit state: every <Z_q>, samples, a measurement with collapse
        {"name": "measure27", "kind": "measure", "dtype": "complex64", "n": 27, "shots": 20000, "qubits": 2},
        # a variational batch of ragged sizes: 600 ansatz circuits of 10 to 20 qubits, 8 strings each
        {"name": "batch600", "kind": "batch", "dtype": "complex64", "n": 20, "nmin": 10, "count": 600, "layers": 6,
         "strings": 8},
    ]


def draw(rng):
    kind = rng.choice(["gates", "gates", "dense", "dense", "fused", "fused", "fused", "energy", "measure", "batch"])
    dtype = rng.choice(["complex64", "complex64", "complex128"])
    wide = dtype == "complex128"
    if kind == "gates":
        n = rng.randint(12, 26 if wide else 28)
        most = 300 if n <= 20 else 78
        return {"kind": kind, "dtype": dtype, "n": n, "gates": int(round(math.exp(rng.uniform(math.log(20), math.log(most))))),
                "two": rng.choice(["cz,cnot", "cz,cnot,crz", "crz"])}
    if kind == "dense":
        k = rng.randint(1, 6)
        return {"kind": kind, "dtype": dtype, "n": rng.randint(14, (26 if k <= 4 else 24) if wide else 28), "k": k,
                "sets": rng.randint(1, 3)}
    if kind == "fused":
        prec = "native" if wide else rng.choice(["native", "tf32", "split_bf16"])
        return {"kind": kind, "dtype": dtype, "n": rng.randint(14, 24 if wide else 27), "form": rng.choice(["layered", "brick"]),
                "layers": rng.randint(2, 5 if wide else 6), "w": rng.randint(2, 4) if wide else rng.randint(3, 6), "prec": prec}
    if kind == "energy":
        return {"kind": kind, "dtype": dtype, "n": rng.randint(14, 26 if wide else 28), "form": rng.choice(["hopping", "random"]),
                "rotations": rng.randint(0, 6), "strings": rng.randint(3, 24)}
    if kind == "measure":
        return {"kind": kind, "dtype": dtype, "n": rng.randint(14, 25 if wide else 27),
                "shots": int(round(math.exp(rng.uniform(math.log(100), math.log(20000))))), "qubits": rng.randint(1, 5)}
    nmin = rng.randint(8, 12)
    return {"kind": kind, "dtype": "complex64", "n": rng.randint(nmin + 3, 20), "nmin": nmin,
            "count": int(round(math.exp(rng.uniform(math.log(32), math.log(600))))), "layers": rng.randint(2, 6),
            "strings": rng.randint(1, 8)}


# ---- inputs, from the seed alone ----

def _dtype(case):
    return torch.complex64 if case["dtype"] == "complex64" else torch.complex128


def _circuit(case, seed):
    n = case["n"]
    if case["kind"] == "gates":
        return gen.layered_random_circuit(n, 1000, seed, tuple(case["two"].split(",")), max_gates=case["gates"])
    if case["form"] == "brick":
        return gen.circuit_config2(n, case["layers"], seed)
    return gen.circuit_config1(n, case["layers"], seed)


def _dense_gates(case, seed):
    rng = gen.rng_for(seed)
    out = []
    for _ in range(case["sets"]):
        targets = tuple(int(q) for q in rng.choice(case["n"], case["k"], replace=False))
        out.append((targets, gen.random_gate_dense(rng, case["k"])))
    return out


def _random_state(case, seed):
    """A random-circuit-like state: complex normal amplitudes, normalised."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    real = torch.float32 if case["dtype"] == "complex64" else torch.float64
    v = torch.randn((1 << case["n"], 2), generator=g, device="cuda", dtype=real)
    v /= torch.linalg.vector_norm(v)
    return torch.view_as_complex(v)


def _product_state(case, seed):
    """Each qubit at a random point of the Bloch sphere: the mean-field start of a time evolution."""
    rng = gen.rng_for(seed)
    psi = torch.ones(1, dtype=_dtype(case), device="cuda")
    for _ in range(case["n"]):
        a, b = rng.uniform(0.15, 1.4), rng.uniform(0, 2 * np.pi)
        one = torch.tensor([np.cos(a), np.sin(a) * np.exp(1j * b)], dtype=torch.complex128).to(psi)
        psi = torch.outer(one, psi).reshape(-1)
    return psi.contiguous()


def _terms(case, seed):
    """Pauli codes (strings, n) of the Hamiltonian's terms and the rotation angles of one Trotter step.
    hopping: for random pairs p < q, X Z...Z X and Y Z...Z Y between them (Jordan-Wigner) and the density term Z_p Z_q;
    random: every site uniform over I, X, Y, Z."""
    rng, n, count = gen.rng_for(seed), case["n"], case["strings"]
    if case["form"] == "random":
        paulis = rng.integers(0, 4, size=(count, n)).astype(np.int32)
    else:
        paulis = np.zeros((count, n), np.int32)
        for s in range(0, count, 3):
            p, q = sorted(int(x) for x in rng.choice(n, 2, replace=False))
            for j, c in enumerate((gen.PAULI_X, gen.PAULI_Y, gen.PAULI_Z)):
                if s + j < count:
                    if c != gen.PAULI_Z:
                        paulis[s + j, p + 1:q] = gen.PAULI_Z
                    paulis[s + j, [p, q]] = c
    return paulis, rng.uniform(0.02, 0.3, size=case["rotations"])


def _batch_states(case, seed):
    rng = gen.rng_for(seed)
    out = []
    for _ in range(case["count"]):
        n = int(rng.integers(case["nmin"], case["n"] + 1))
        gates = gen.ansatz_circuit(n, case["layers"], rng)
        out.append((n, gates, gen.random_pauli_strings(n, case["strings"], rng)[0]))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        b = sv.Batch(torch.cuda.current_stream())
        b.compile(_batch_states(case, seed))
        return {"case": case, "batch": b, "buf": torch.empty(b.state_amps, dtype=torch.complex64, device="cuda")}
    if kind in ("gates", "fused"):
        psi = torch.zeros(1 << case["n"], dtype=_dtype(case), device="cuda")
    else:
        psi = _product_state(case, seed) if kind == "energy" else _random_state(case, seed)
    st = {"case": case, "psi": psi, "sv": sv.StateVector(psi)}
    if kind in ("gates", "fused"):
        st["gates"] = _circuit(case, seed)
    elif kind == "dense":
        st["gates"] = _dense_gates(case, seed)
    elif kind == "energy":
        st["paulis"], st["angles"] = _terms(case, seed)
        st["sites"] = np.tile(np.arange(case["n"], dtype=np.int32), (case["strings"], 1))
    else:
        rng = gen.rng_for(seed)
        st["rands"], st["outcome"] = rng.random(case["shots"]), float(rng.random())
        st["qubits"] = [int(q) for q in rng.choice(case["n"], case["qubits"], replace=False)]
    return st


# ---- one pass ----

def _values(case, x):
    return np.asarray(x, dtype=np.float32 if case["dtype"] == "complex64" else np.float64)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        state["batch"].launch(state["buf"])
        return _values(case, np.concatenate(state["batch"].results()))
    s, psi = state["sv"], state["psi"]
    if kind == "gates":
        s.set_basis_state(0)
        s.apply_circuit(state["gates"])
        return {"state": psi, "parity": _values(case, s.measure_probs(range(case["n"])))}
    if kind == "dense":
        for targets, matrix in state["gates"]:
            s.apply(targets, matrix)
        return psi
    if kind == "fused":
        s.set_basis_state(0)
        s.apply_fused(state["gates"], case["w"], PREC[case["prec"]])
        return psi
    if kind == "energy":
        for i, theta in enumerate(state["angles"]):
            j = i % case["strings"]
            s.pauli_rotation(theta, state["paulis"][j], state["sites"][j])
        return {"state": psi, "terms": _values(case, s.expectation_pauli(state["paulis"], state["sites"]))}
    z = s.expectation_z_all()
    samples = s.sample(state["rands"])
    parity = s.measure(state["qubits"], state["outcome"], collapse=True)
    return {"z": _values(case, z), "samples": samples, "parity": parity, "state": psi}


# ---- what a pass cannot do without ----

def _gate_share(g):
    """Share of the amplitudes that a gate has to touch: the half or quarter that a control or a CZ leaves."""
    if g.name == "cz":
        return 0.25
    return 0.5 if g.controls else 1.0


def work(case):
    n, kind = case["n"], case["kind"]
    size = 8 if case["dtype"] == "complex64" else 16
    amps = float(1 << n)
    if kind == "batch":
        ns = range(case["nmin"], n + 1)
        mean = sum(m * 2.0 ** m for m in ns) / len(ns)          # qubits x amplitudes of the average state
        flops = case["count"] * case["layers"] * mean * 16
        return {"bytes": 8.0 * case["count"] * case["strings"], "flops": flops}
    if kind in ("gates", "fused"):
        gates = _circuit(case, 1)
        flops = sum(amps * (14 if g.name == "su2" else 6 * _gate_share(g) if g.name == "crz" else 0) for g in gates)
        if kind == "fused":
            return {"bytes": amps * size, "flops": flops}
        return {"bytes": amps * size * (2 + 2 * sum(_gate_share(g) for g in gates)), "flops": flops}
    if kind == "dense":
        return {"bytes": 2 * amps * size * case["sets"], "flops": 8.0 * (1 << case["k"]) * amps * case["sets"]}
    if kind == "energy":
        return {"bytes": amps * size * (2 * case["rotations"] + 1),
                "flops": amps * (8 * case["rotations"] + 4 * case["strings"])}
    # <Z_q> and the samples share nothing: each reads the state; the collapse reads half of it and writes all of it
    return {"bytes": amps * size * (1 + 1 + 1 + 1.5), "flops": amps * (4 + 3 + 3 + n)}


# ---- the same in 64 bits with plain torch ----

def _apply(psi, targets, matrix, controls=(), cvals=()):
    """matrix on the targets (bit j of its index is targets[j]) where the controls hold, in place."""
    n = psi.numel().bit_length() - 1
    qs = sorted([*targets, *controls], reverse=True)
    shape, at = [], n
    for q in qs:
        shape += [1 << (at - q - 1), 2]
        at = q
    v = psi.view(shape + [1 << at])
    axis = {q: 2 * i + 1 for i, q in enumerate(qs)}
    index = [slice(None)] * v.dim()
    for q, b in zip(controls, cvals):
        index[axis[q]] = slice(b, b + 1)
    v = v[tuple(index)]
    front = v.movedim([axis[q] for q in reversed(targets)], list(range(len(targets))))
    m = torch.as_tensor(np.asarray(matrix), dtype=torch.complex128, device=psi.device)
    new = m @ front.reshape(m.shape[0], -1)
    front.copy_(new.view(front.shape))


def _apply_all(psi, gates):
    for g in gates:
        cv = tuple(g.control_values) if g.control_values else (1,) * len(g.controls)
        _apply(psi, tuple(g.targets), g.matrix, tuple(g.controls), cv)


def _pauli(psi, codes):
    """P psi for one string of Pauli codes, a new tensor."""
    out = psi
    for q, c in enumerate(codes):
        if c == 0:
            continue
        v = out.view(-1, 2, 1 << q)
        if c == gen.PAULI_Z:
            out = torch.stack([v[:, 0], -v[:, 1]], 1).reshape(-1)
        elif c == gen.PAULI_X:
            out = torch.stack([v[:, 1], v[:, 0]], 1).reshape(-1)
        else:
            out = torch.stack([-1j * v[:, 1], 1j * v[:, 0]], 1).reshape(-1)
    return out


def _signed(p, q):
    v = p.view(-1, 2, 1 << q)
    return torch.stack([v[:, 0], -v[:, 1]], 1).reshape(-1)


def _exact_batch(case, seed):
    states = _batch_states(case, seed)
    out = [None] * len(states)
    for n in sorted({s[0] for s in states}):
        ids = [i for i, s in enumerate(states) if s[0] == n]
        for lo in range(0, len(ids), 128):
            part = ids[lo:lo + 128]
            psi = torch.zeros((len(part), 1 << n), dtype=torch.complex128, device="cuda")
            psi[:, 0] = 1
            for g, first in enumerate(states[part[0]][1]):   # circuits of one size differ in their angles only
                t = first.targets[0]
                if first.controls:
                    c = first.controls[0]
                    index = torch.arange(1 << n, device="cuda")
                    psi = psi[:, torch.where((index >> c) & 1 == 1, index ^ (1 << t), index)]
                else:
                    m = torch.as_tensor(np.stack([states[i][1][g].matrix for i in part]), device="cuda")
                    v = psi.view(len(part), -1, 2, 1 << t)
                    psi = torch.einsum("sab,sxbl->sxal", m, v).reshape(len(part), -1)
            for row, i in enumerate(part):
                out[i] = [float(torch.vdot(psi[row], _pauli(psi[row], codes)).real) for codes in states[i][2]]
    return np.concatenate(out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind in ("gates", "fused"):
        psi = torch.zeros(1 << case["n"], dtype=torch.complex128, device="cuda")
        psi[0] = 1
        _apply_all(psi, _circuit(case, seed))
        if kind == "fused":
            return psi
        p = psi.abs().square()
        for q in range(case["n"]):   # +p where the parity of the low qubits is even, -p where it is odd
            p = _signed(p, q)
        d, t = float(p.sum()), float(psi.abs().square().sum())
        return {"state": psi, "parity": np.array([(t + d) / 2, (t - d) / 2])}
    if kind == "dense":
        psi = _random_state(case, seed).to(torch.complex128)
        for targets, matrix in _dense_gates(case, seed):
            _apply(psi, targets, matrix)
        return psi
    if kind == "energy":
        psi = _product_state(case, seed).to(torch.complex128)
        paulis, angles = _terms(case, seed)
        for i, theta in enumerate(angles):
            psi = math.cos(theta) * psi + 1j * math.sin(theta) * _pauli(psi, paulis[i % case["strings"]])
        return {"state": psi, "terms": np.array([float(torch.vdot(psi, _pauli(psi, c)).real) for c in paulis])}
    psi = _random_state(case, seed).to(torch.complex128)
    rng = gen.rng_for(seed)
    rng.random(case["shots"])
    outcome = float(rng.random())
    qubits = [int(q) for q in rng.choice(case["n"], case["qubits"], replace=False)]
    p = psi.abs().square()
    z = np.array([float(_signed(p, q).sum()) for q in range(case["n"])])
    s = p
    for q in qubits:
        s = _signed(s, q)
    t, d = float(p.sum()), float(s.sum())
    even, odd = (t + d) / 2, (t - d) / 2
    parity = 0 if outcome < even / (even + odd) else 1
    sign = torch.ones_like(p)
    for q in qubits:
        sign = _signed(sign, q)
    psi = torch.where(sign > 0 if parity == 0 else sign < 0, psi / math.sqrt(even if parity == 0 else odd), 0)
    return {"z": z, "samples": None, "parity": None, "state": psi}
