"""The work that users of the simulator have it do, as cases that can be timed.

A case is a dict of plain values.  Its "kind" says which public calls it makes:

* circuit: a planned circuit executed on a state in device memory
  (``StateVector.plan`` / ``Plan.execute``), complex64 or complex128, in the
  tiled or the per-gate mode;
* blocks: dense k-qubit operators applied one after another
  (``StateVector.apply_fused``);
* code: the two-byte amplitude code: a complex64 state is encoded, a circuit
  runs on the codes, the result is decoded (``encode_from``, ``Plan.execute``,
  ``decode_to``);
* readout: the observables of a state: <sigma^x,y,z> of every qubit, the norm
  and 1024 chosen amplitudes;
* cut: amplitudes of a grid circuit by the decomposition of the gates across
  its middle (``sv_cut_amplitudes``);
* batch: independent circuits of different sizes together (``Batch``).

The circuit of a case is fixed by the case (a user plans a circuit once); the
state it acts on, the operators, the bit strings and the indices come from the
seed.  States are complex Gaussian, normalised, which is what the amplitudes of
a random circuit look like.
"""

import functools
import math

import numpy as np
import torch

from paper_1912_03243_gb300 import circuits as C
from paper_1912_03243_gb300 import sv

DEV = "cuda"


def listed():
    return [
        # a small register run many times (parameter scans, teaching, tests): launches and latency count
        {"name": "random_10q_c64", "kind": "circuit", "family": "random", "n": 10, "depth": 10, "dtype": "c64", "mode": "tiled"},
        # a register of a few tiles, an odd qubit count: too little work to fill the chip
        {"name": "random_17q_c64", "kind": "circuit", "family": "random", "n": 17, "depth": 12, "dtype": "c64", "mode": "tiled"},
        # an everyday simulation: the 24-qubit instance the tests check against the oracle
        {"name": "random_24q_c64", "kind": "circuit", "family": "random", "n": 24, "depth": 16, "dtype": "c64", "mode": "tiled"},
        # the large simulation: the 30-qubit random circuit of the benchmark
        {"name": "random_30q_c64", "kind": "circuit", "family": "random", "n": 30, "depth": 16, "dtype": "c64", "mode": "tiled"},
        # an algorithm circuit: controlled phases and swaps, an odd qubit count
        {"name": "qft_27q_c64", "kind": "circuit", "family": "qft", "n": 27, "depth": 1, "dtype": "c64", "mode": "tiled"},
        # the reference-precision run gate by gate (20 qubits, depth 20)
        {"name": "pergate_20q_c128", "kind": "circuit", "family": "random", "n": 20, "depth": 20, "dtype": "c128", "mode": "pergate"},
        # the reference precision on a larger register, in passes of many gates
        {"name": "random_25q_c128", "kind": "circuit", "family": "random", "n": 25, "depth": 8, "dtype": "c128", "mode": "tiled"},
        # the two-byte code: the memory-saving run of a register that would not fit otherwise (here at 27 qubits)
        {"name": "code_27q", "kind": "code", "n": 27, "depth": 4},
        # dense operators on a few qubits (compiled blocks, Trotter steps), low, high and mixed qubits
        {"name": "blocks_27q_c64", "kind": "blocks", "n": 27, "dtype": "c64", "kmax": 6, "count": 6},
        # what is read from a state after a run
        {"name": "readout_28q_c64", "kind": "readout", "n": 28, "dtype": "c64"},
        # a 48-qubit grid circuit cut into two halves: 256 branches
        {"name": "cut_6x8_d8", "kind": "cut", "rows": 6, "cols": 8, "depth": 8, "m": 1024},
        # many unrelated circuits of different sizes at once
        {"name": "batch_64", "kind": "batch", "count": 64, "nmin": 13, "nmax": 22, "depth": 10},
    ]


def draw(rng):
    kind = rng.choice(["circuit", "circuit", "circuit", "blocks", "code", "code", "readout", "cut", "batch"])
    cseed = rng.randrange(1, 1 << 20)
    if kind == "circuit":
        mode, dtype = rng.choice([("tiled", "c64"), ("tiled", "c64"), ("tiled", "c128"), ("pergate", "c64"), ("pergate", "c128")])
        n = rng.randint(6, {("tiled", "c64"): 29, ("tiled", "c128"): 25, ("pergate", "c64"): 26, ("pergate", "c128"): 25}[mode, dtype])
        family = rng.choice(["random", "random", "mixed", "qft"])
        return {"kind": kind, "family": family, "n": n, "depth": rng.randint(3, 16 if mode == "tiled" else 8), "dtype": dtype, "mode": mode, "cseed": cseed}
    if kind == "blocks":
        dtype = rng.choice(["c64", "c64", "c128"])
        return {"kind": kind, "n": rng.randint(7, 28 if dtype == "c64" else 23), "dtype": dtype, "kmax": rng.randint(1, 6), "count": rng.randint(1, 8), "cseed": cseed}
    if kind == "code":
        return {"kind": kind, "n": rng.randint(5, 28), "depth": rng.randint(1, 6), "cseed": cseed}
    if kind == "readout":
        dtype = rng.choice(["c64", "c128", "code"])
        return {"kind": kind, "n": rng.randint(3, 28 if dtype != "c128" else 26), "dtype": dtype, "cseed": cseed}
    if kind == "cut":
        while True:
            rows, cols, depth = rng.randint(3, 6), rng.randint(3, 8), rng.randint(3, 9)
            if 12 <= rows * cols <= 48 and _cut_work(rows, cols, depth) <= 1 << 32:
                return {"kind": kind, "rows": rows, "cols": cols, "depth": depth, "m": rng.choice([1, 100, 1024, 3001]), "cseed": cseed}
    lo = rng.randint(8, 16)
    return {"kind": kind, "count": rng.randint(3, 64), "nmin": lo, "nmax": rng.randint(lo, 20), "depth": rng.randint(2, 10), "cseed": cseed}


# ---- the circuits of a case

@functools.lru_cache(maxsize=None)
def _circuit(family, n, depth, cseed):
    if family == "qft":
        return C.qft_circuit(n)
    if family == "mixed":  # every gate kind of the text format on random qubits
        return C.random_unitary_gates(n, depth * n, cseed)
    return C.random_circuit(n, depth, cseed)


def _case_circuit(case):
    return _circuit(case["family"], case["n"], case["depth"], case.get("cseed", 1))


def _grid(case):
    rows, cols = case["rows"], case["cols"]
    return C.grid_circuit(rows, cols, case["depth"], case.get("cseed", 1)), rows * cols, C.grid_partition_mask(rows, cols, rows // 2)


def _cut_gates(rows, cols, depth):
    half = (rows // 2) * cols
    return sum((a < half) != (b < half) for layer in range(depth) for a, b in C.grid_edges(rows, cols, C.GRID_PATTERNS[layer % 6]))


def _cut_work(rows, cols, depth):
    """Amplitudes of all branches of both halves."""
    a = (rows // 2) * cols
    return ((1 << a) + (1 << (rows * cols - a))) << _cut_gates(rows, cols, depth)


def _members(case):
    r = np.random.Generator(np.random.PCG64(case.get("cseed", 64)))
    ns = [int(v) for v in r.integers(case["nmin"], case["nmax"] + 1, size=case["count"])]
    return [(n, C.random_circuit(n, case["depth"], 500 + k)) for k, n in enumerate(ns)]


def _blocks(case, seed):
    """Qubit lists of the dense operators: low, high and random qubits, widths up to kmax."""
    r = np.random.Generator(np.random.PCG64(case.get("cseed", 5)))
    n, kmax = case["n"], min(case["kmax"], case["n"])
    u = np.random.Generator(np.random.PCG64(seed))
    out = []
    for i in range(case["count"]):
        k = max(1, kmax - i // 3)
        q = list(range(k)) if i % 3 == 0 else list(range(n - k, n)) if i % 3 == 1 else [int(v) for v in r.choice(n, size=k, replace=False)]
        z = u.normal(size=(1 << k, 1 << k)) + 1j * u.normal(size=(1 << k, 1 << k))
        out.append((q, np.linalg.qr(z)[0]))
    return out


# ---- states

def _random_into(out, seed):
    """Fill a complex tensor with a normalised Gaussian state."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    flat = torch.view_as_real(out).reshape(-1)
    step = 1 << 28
    for i in range(0, flat.numel(), step):
        flat[i:i + step].normal_(generator=g)
    total = sum(float(flat[i:i + step].double().square().sum()) for i in range(0, flat.numel(), step))
    flat.mul_(1.0 / math.sqrt(total))


def _amps(s):
    """The amplitudes of a state as a complex tensor (its own memory)."""
    return s.buffer.view(torch.complex64 if s.dtype == "c64" else torch.complex128)


def _state(n, dtype, seed):
    s = sv.StateVector(n, dtype)
    _random_into(_amps(s), seed)
    return s


def _code_parts(s):
    n = s.n
    return {"codes": s.buffer[: 2 << n].view(torch.int8), "scales": s.buffer[2 << n:].view(torch.float32)}


# ---- the cases

def prepare(case, seed):
    kind = case["kind"]
    if kind == "circuit":
        s = _state(case["n"], case["dtype"], seed)
        return {"kind": kind, "s": s, "plan": s.plan(_case_circuit(case), case["mode"])}
    if kind == "blocks":
        return {"kind": kind, "s": _state(case["n"], case["dtype"], seed), "blocks": _blocks(case, seed)}
    if kind == "code":
        src = _state(case["n"], "c64", seed)
        enc, dst = sv.StateVector(case["n"], "enc2b"), sv.StateVector(case["n"], "c64")
        return {"kind": kind, "src": src, "enc": enc, "dst": dst, "plan": enc.plan(_circuit("random", case["n"], case["depth"], case.get("cseed", 1)), "pergate")}
    if kind == "readout":
        s = _state(case["n"], "c64" if case["dtype"] == "code" else case["dtype"], seed)
        if case["dtype"] == "code":
            e = sv.StateVector(case["n"], "enc2b")
            e.encode_from(s)
            s = e
        return {"kind": kind, "s": s, "idx": C.random_bitstrings(1024, case["n"], seed)}
    if kind == "cut":
        c, n, mask = _grid(case)
        return {"kind": kind, "c": c, "n": n, "mask": mask, "z": C.random_bitstrings(case["m"], n, seed)}
    mem = _members(case)
    states = [_state(n, "c64", seed * 1000 + k) for k, (n, _) in enumerate(mem)]
    return {"kind": kind, "states": states, "batch": sv.Batch(states, [c for _, c in mem])}


def run(st):
    kind = st["kind"]
    if kind == "circuit":
        st["plan"].execute()
        return _amps(st["s"])
    if kind == "blocks":
        for q, u in st["blocks"]:
            st["s"].apply_fused(q, u)
        return _amps(st["s"])
    if kind == "code":
        st["enc"].encode_from(st["src"])
        st["plan"].execute()
        st["enc"].decode_to(st["dst"])
        return {**_code_parts(st["enc"]), "decoded": _amps(st["dst"])}
    if kind == "readout":
        s = st["s"]
        return {"sigma": s.expect_pauli(), "norm": s.norm(), "amplitudes": s.amplitudes(st["idx"])}
    if kind == "cut":
        return sv.sv_cut_amplitudes(st["c"], st["n"], st["mask"], st["z"])[0]
    st["batch"].execute()
    return [_amps(s) for s in st["states"]]


# ---- what a pass cannot do without

_ADDS = {"T": 1, "TDG": 1, "S": 0, "SDG": 0, "X": 0, "Y": 0, "Z": 0, "CZ": 0, "CX": 0, "SWAP": 0, "P": 2, "CP": 1, "U": 8}


def _circuit_flops(c, amps):
    """Real operations per amplitude: 2 for a butterfly (H, SX, SY and their
    adjoints), 1 for an eighth-turn phase, signs and permutations free."""
    return float(amps) * sum(_ADDS.get(g[0], 2) for g in c.gates)


def work(case):
    kind = case["kind"]
    size = {"c64": 8, "c128": 16, "code": 2}[case.get("dtype", "c64")]
    if kind == "circuit":
        return {"bytes": 2.0 * size * (1 << case["n"]), "flops": _circuit_flops(_case_circuit(case), 1 << case["n"])}
    if kind == "blocks":
        ks = [len(q) for q, _ in _blocks(case, 0)]
        return {"bytes": 2.0 * size * (1 << case["n"]) * len(ks), "flops": sum(8.0 * (1 << k) for k in ks) * (1 << case["n"])}
    if kind == "code":
        c = _circuit("random", case["n"], case["depth"], case.get("cseed", 1))
        return {"bytes": (8.0 + 2.0 + 2.0 + 2.0 + 8.0) * (1 << case["n"]), "flops": _circuit_flops(c, 1 << case["n"])}
    if kind == "readout":  # <x>, <y>: 8 operations per pair and qubit; the probabilities: 4 per amplitude
        return {"bytes": 1.0 * size * (1 << case["n"]) + 24 * 1024, "flops": (4.0 * case["n"] + 4.0) * (1 << case["n"])}
    if kind == "cut":
        amps = _cut_work(case["rows"], case["cols"], case["depth"])
        return {"bytes": 24.0 * case["m"], "flops": 2.0 * amps}  # each branch amplitude once in the products
    mem = _members(case)
    return {"bytes": sum(16.0 * (1 << n) for n, _ in mem), "flops": sum(_circuit_flops(c, 1 << n) for n, c in mem)}


# ---- the same in 64 bits, plainly

_R = math.sqrt(0.5)
_P, _M = 0.5 + 0.5j, 0.5 - 0.5j
_GATES = {
    "H": [[_R, _R], [_R, -_R]], "X": [[0, 1], [1, 0]], "Y": [[0, -1j], [1j, 0]], "Z": [[1, 0], [0, -1]],
    "S": [[1, 0], [0, 1j]], "SDG": [[1, 0], [0, -1j]], "T": [[1, 0], [0, complex(_R, _R)]], "TDG": [[1, 0], [0, complex(_R, -_R)]],
    "SX": [[_P, _M], [_M, _P]], "SXDG": [[_M, _P], [_P, _M]], "SY": [[_P, -_P], [_P, _P]], "SYDG": [[_M, _M], [-_M, _M]],
}


def _apply_1q(psi, q, u, where=None):
    """Update the pairs of bit q (of the half where bit `where` is set) in place."""
    n = psi.numel().bit_length() - 1
    bits = sorted([q] if where is None else [q, where], reverse=True)
    shape, last = [], n
    for b in bits:
        shape += [1 << (last - 1 - b), 2]
        last = b
    v = psi.view(shape + [1 << last])
    at = [slice(None)] * v.dim()
    if where is not None:
        at[2 * bits.index(where) + 1] = 1
    lo, hi = list(at), list(at)
    lo[2 * bits.index(q) + 1], hi[2 * bits.index(q) + 1] = 0, 1
    a, b = v[tuple(lo)], v[tuple(hi)]
    u = [[complex(x) for x in row] for row in u]
    if u[0][1] == 0 and u[1][0] == 0:
        for x, f in ((a, u[0][0]), (b, u[1][1])):
            if f != 1:
                x.mul_(f)
        return
    na = a * u[0][0]
    na.add_(b, alpha=u[0][1])
    nb = b * u[1][1]
    nb.add_(a, alpha=u[1][0])
    a.copy_(na)
    b.copy_(nb)


def _apply(psi, gate):
    name, q, p = gate
    if name == "CZ":
        _apply_1q(psi, q[1], _GATES["Z"], q[0])
    elif name == "CX":
        _apply_1q(psi, q[1], _GATES["X"], q[0])
    elif name == "CP":
        _apply_1q(psi, q[1], [[1, 0], [0, complex(math.cos(p[0]), math.sin(p[0]))]], q[0])
    elif name == "SWAP":
        for a, b in ((q[0], q[1]), (q[1], q[0]), (q[0], q[1])):
            _apply_1q(psi, b, _GATES["X"], a)
    elif name == "P":
        _apply_1q(psi, q[0], [[1, 0], [0, complex(math.cos(p[0]), math.sin(p[0]))]])
    elif name == "U":
        _apply_1q(psi, q[0], [[complex(p[0], p[1]), complex(p[2], p[3])], [complex(p[4], p[5]), complex(p[6], p[7])]])
    else:
        _apply_1q(psi, q[0], _GATES[name])


def _run_exact(psi, c):
    for g in c.gates:
        _apply(psi, g)
    return psi


def _start_state(n, dtype, seed):
    psi = torch.empty(1 << n, dtype=torch.complex64 if dtype == "c64" else torch.complex128, device=DEV)
    _random_into(psi, seed)
    return psi.to(torch.complex128)


def _sigma_exact(psi, n):
    out = torch.zeros(n, 3, dtype=torch.float64)
    prob = torch.view_as_real(psi).square().sum(-1)
    for q in range(n):
        v = psi.view(-1, 2, 1 << q)
        ov = (v[:, 0].conj() * v[:, 1]).sum()
        z = prob.view(-1, 2, 1 << q).sum((0, 2))
        out[q] = torch.tensor([2 * float(ov.real), 2 * float(ov.imag), float(z[0] - z[1])])
    return out.numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind == "circuit":
        c = _case_circuit(case)
        if len(c) << case["n"] > 700 << 27:
            return None
        return _run_exact(_start_state(case["n"], case["dtype"], seed), c)
    if kind == "blocks":
        psi = _start_state(case["n"], case["dtype"], seed)
        n = case["n"]
        for q, u in _blocks(case, seed):
            k = len(q)
            axes = [n - 1 - b for b in reversed(q)]  # most significant local bit first
            v = psi.view([2] * n).movedim(axes, list(range(k)))
            shape = v.shape
            v = (torch.from_numpy(u).to(DEV) @ v.reshape(1 << k, -1)).view(shape)
            psi = v.movedim(list(range(k)), axes).reshape(-1)
        return psi
    if kind == "readout" and case["dtype"] != "code":
        psi = _start_state(case["n"], case["dtype"], seed)
        idx = torch.from_numpy(C.random_bitstrings(1024, case["n"], seed).astype(np.int64)).to(DEV)
        return {"sigma": _sigma_exact(psi, case["n"]), "norm": float(torch.view_as_real(psi).square().sum()), "amplitudes": psi[idx].cpu().numpy()}
    if kind == "cut":
        c, n, _ = _grid(case)
        if len(c) << n > 700 << 27 or n > 28:
            return None
        psi = torch.zeros(1 << n, dtype=torch.complex128, device=DEV)
        psi[0] = 1
        _run_exact(psi, c)
        return psi[torch.from_numpy(C.random_bitstrings(case["m"], n, seed).astype(np.int64)).to(DEV)].cpu().numpy()
    if kind == "batch":
        return [_run_exact(_start_state(n, "c64", seed * 1000 + k), c) for k, (n, c) in enumerate(_members(case))]
    return None
