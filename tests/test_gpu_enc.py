"""GPU two-byte code against the CPU codec mirror: codes and scales must be
bit-exact (integer/byte work); fidelity against the exact oracle is
measured and reported."""

import math

import numpy as np
import pytest

from paper_1912_03243_gb300 import circuits as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_03243_gb300 import build, sv

    build.build()
    sv.lib()
    return sv


def raw_of(codes, scales):
    return np.concatenate([codes.view(np.uint8), scales.view(np.uint8)])


def split_raw(raw, n):
    codes = raw[: 2 << n].view(np.int8)
    scales = raw[2 << n:].view(np.float32)
    return codes, scales


def rand_c64(n, seed, zero_block=True):
    rng = np.random.default_rng(seed)
    psi = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)).astype(np.complex64)
    if zero_block and n >= 9:
        psi[256:512] = 0
    return psi


@pytest.mark.parametrize("n", [1, 3, 7, 8, 9, 12])
def test_encode_decode_bit_exact(S, orc, n):
    psi = rand_c64(n, n)
    src = S.StateVector(n, "c64")
    src.from_numpy(psi)
    enc = S.StateVector(n, "enc2b")
    enc.encode_from(src)
    codes, scales = enc.codes()
    rc, rs = orc.enc_encode(psi)
    assert np.array_equal(codes, rc)
    assert np.array_equal(scales.view(np.uint32), rs.view(np.uint32))
    dst = S.StateVector(n, "c64")
    enc.decode_to(dst)
    got = dst.to_numpy()
    ref = orc.enc_decode(rc, rs)
    assert np.array_equal(got.view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("n", [4, 10])
def test_gate_every_target_control_bit_exact(S, orc, n):
    psi = rand_c64(n, 77 + n)
    codes, scales = orc.enc_encode(psi)
    enc = S.StateVector(n, "enc2b")
    mats = [orc.gate_matrix(k) for k in ("H", "SX", "SY", "T", "X", "Z")]
    rng = np.random.default_rng(n)
    z = rng.normal(size=(2, 2)) + 1j * rng.normal(size=(2, 2))
    mats.append(np.linalg.qr(z)[0])
    mats.append(np.diag([1.0, np.exp(0.3j)]))  # a phase (u00 = 1) other than T
    for u in mats:
        for t in range(n):
            for c in [-1] + [q for q in range(n) if q != t]:
                enc.from_numpy(raw_of(codes, scales))
                enc.apply_gate(t, u, control=c)
                gc, gs = enc.codes()
                rc, rs = orc.enc_apply_gate(codes, scales, t, c, u)
                assert np.array_equal(gc, rc), (t, c)
                assert np.array_equal(gs.view(np.uint32), rs.view(np.uint32)), (t, c)


@pytest.mark.parametrize("n,depth,seed", [(6, 6, 1), (16, 8, 2), (18, 12, 3)])
def test_random_circuit_bit_exact(S, orc, n, depth, seed):
    c = C.random_circuit(n, depth, seed)
    rc, rs = orc.enc_run(c)
    enc = S.StateVector(n, "enc2b")
    enc.run(c, "pergate")
    gc, gs = enc.codes()
    assert np.array_equal(gc, rc)
    assert np.array_equal(gs.view(np.uint32), rs.view(np.uint32))


def test_qft_and_ghz_bit_exact(S, orc):
    n = 12
    for c in (C.qft_circuit(n, 0x5A5), C.ghz_circuit(n)):
        rc, rs = orc.enc_run(c)
        enc = S.StateVector(n, "enc2b")
        enc.run(c)
        gc, gs = enc.codes()
        assert np.array_equal(gc, rc) and np.array_equal(gs, rs)


def test_uniform_exact_large(S):
    """Sec. 3: the code represents the uniform superposition exactly (all
    codes 127), here at 28 qubits."""
    n = 28
    enc = S.StateVector(n, "enc2b")
    enc.run(C.uniform_circuit(n))
    codes, scales = enc.codes()
    assert np.all(codes[0::2] == 127) and np.all(codes[1::2] == 0)
    assert np.all(scales == scales[0])
    nrm = enc.norm()
    assert abs(nrm / ((1 << n) * float(scales[0]) ** 2) - 1) < 1e-12


def test_fidelity_24q(S, orc, record_property):
    """Fidelity of the encoded simulation against the FP64 oracle on a
    24-qubit instance of the depth-12 random circuit (measured, reported)."""
    n = 24
    c = C.random_circuit(n, 12, 1)
    exact = orc.run(c)
    enc = S.StateVector(n, "enc2b")
    enc.run(c)
    dec = S.StateVector(n, "c64")
    enc.decode_to(dec)
    got = dec.to_numpy().astype(np.complex128)
    f = abs(np.vdot(exact, got)) ** 2 / (np.vdot(exact, exact).real * np.vdot(got, got).real)
    record_property("fidelity_enc2b_24q_d12", f)
    print(f"enc2b fidelity 24q d12: {f:.6f}")
    assert f > 0.95


@pytest.mark.parametrize("n,seed", [(9, 1), (12, 2), (14, 3)])
def test_in_block_runs_bit_exact(S, orc, n, seed):
    """Runs of consecutive in-block gates and sign flips applied in one pass
    each (the default per-gate plan of the two-byte code) give the CPU codec
    mirror's codes: every gate kind of the format on random qubits, so runs
    hold controls inside and outside the blocks, X, P, U and CZ/CP flips, and
    runs are broken by gates across blocks."""
    c = C.random_unitary_gates(n, 400, 50 + seed)
    layer_like = C.random_circuit(n, 8, seed)  # long runs: in-block layers and CZ rows
    for circ in (c, layer_like):
        rc, rs = orc.enc_run(circ)
        enc = S.StateVector(n, "enc2b")
        plan = enc.plan(circ, "pergate")
        kinds = {name for name, _ in plan.launch_info()}
        plan.execute()
        gc, gs = enc.codes()
        assert np.array_equal(gc, rc), n
        assert np.array_equal(gs.view(np.uint32), rs.view(np.uint32)), n
        plan.free()
    assert "k_enc_run_in" in kinds


def test_in_block_runs_equal_one_pass_per_gate(S, monkeypatch):
    """At 22 qubits (beyond the mirror's quick range) the fused runs and one
    pass per gate (SV_ENC_RUNS=0) write the same codes and scales."""
    n = 22
    c = C.random_circuit(n, 6, 8)
    out = []
    for runs in ("1", "0"):
        monkeypatch.setenv("SV_ENC_RUNS", runs)
        enc = S.StateVector(n, "enc2b")
        enc.run(c, "pergate")
        out.append(enc.codes())
        enc.free()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1].view(np.uint32), out[1][1].view(np.uint32))


def _mixed_on(n, qubits, count, seed):
    """A mixed circuit (every gate kind) whose gates act on the given qubits of an n-qubit register."""
    small = C.random_unitary_gates(len(qubits), count, seed)
    c = C.Circuit(n)
    for name, qs, ps in small.gates:
        c.add(name, *(qubits[q] for q in qs), params=ps)
    return c


@pytest.mark.parametrize("n,blockq", [(8, []), (9, [8]), (12, [9, 11]), (17, [10, 16]), (20, [8, 19]), (21, [8, 14, 20]),
                                      (22, [9, 13, 18, 21]), (23, [8, 9, 10, 22]), (23, [11, 12, 13, 14, 15])])
def test_runs_across_blocks_bit_exact(S, orc, monkeypatch, n, blockq):
    """Runs that hold gates across blocks (tiles of 1 to 16 blocks, more target
    bits than one tile takes, X on blocks, controls inside and outside the
    blocks and the tile) write the codes of one pass per gate, and at small n
    those of the CPU codec mirror."""
    circs = [_mixed_on(n, [0, 1, 2, 4, 7] + blockq, 150, n), C.random_unitary_gates(n, 60, 9 + n)]
    psi = rand_c64(n, 5)
    src = S.StateVector(n, "c64")
    src.from_numpy(psi)
    for circ in circs:
        out = []
        for runs in ("1", "0"):
            monkeypatch.setenv("SV_ENC_RUNS", runs)
            enc = S.StateVector(n, "enc2b")
            enc.encode_from(src)
            p = enc.plan(circ, "pergate")
            if runs == "1":
                assert p.passes < p.gates
            p.execute()
            p.free()
            out.append(enc.codes())
            enc.free()
        assert np.array_equal(out[0][0], out[1][0])
        assert np.array_equal(out[0][1].view(np.uint32), out[1][1].view(np.uint32))
        if n <= 17:
            rc, rs = orc.enc_run(circ, None, *orc.enc_encode(psi))
            assert np.array_equal(out[0][0], rc)
            assert np.array_equal(out[0][1].view(np.uint32), rs.view(np.uint32))


@pytest.mark.parametrize("n,blockq", [(8, []), (9, []), (16, []), (23, []), (23, [12]), (24, [9, 20])])
def test_runs_with_few_block_bits(S, monkeypatch, n, blockq):
    """Runs inside single blocks (controls outside them too) and runs whose
    tiles are made whole by block bits that no gate targets write the codes of
    one pass per gate."""
    circ = _mixed_on(n, [0, 1, 2, 5, 7] + blockq, 200, n)
    if n > 8:
        for q in (0, 3, 7):
            circ.add("CX", n - 1, q)
            circ.add("H", q)
    psi = rand_c64(n, 6)
    src = S.StateVector(n, "c64")
    src.from_numpy(psi)
    out = []
    for runs in ("1", "0"):
        monkeypatch.setenv("SV_ENC_RUNS", runs)
        enc = S.StateVector(n, "enc2b")
        enc.encode_from(src)
        enc.run(circ, "pergate")
        out.append(enc.codes())
        enc.free()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1].view(np.uint32), out[1][1].view(np.uint32))


def test_runs_inside_blocks_do_their_work_once(S, monkeypatch):
    """A run of gates inside the blocks exists to save passes: at 24 qubits it
    takes no longer than one and a half times those passes (it took almost
    three times as long when every block was computed twice)."""
    import torch

    n = 24
    circ = C.Circuit(n)
    for k in range(48):
        circ.add(("H", "SX", "T", "SY")[k % 4], k % 8)
    ms = {}
    for runs in ("1", "0"):
        monkeypatch.setenv("SV_ENC_RUNS", runs)
        enc = S.StateVector(n, "enc2b")
        p = enc.plan(circ, "pergate")
        ms[runs] = 1e9
        for _ in range(6):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            ev[0].record()
            for _ in range(3):
                p.execute()
            ev[1].record()
            torch.cuda.synchronize()
            ms[runs] = min(ms[runs], ev[0].elapsed_time(ev[1]))
        p.free()
        enc.free()
    assert ms["1"] <= 1.5 * ms["0"], ms


@pytest.mark.parametrize("n", [9, 12, 23, 27])
def test_runs_where_they_are_faster(S, n):
    """A few gates that only move or negate codes keep passes of their own (a
    run decodes the code and computes in its tiles); gates that compute, and
    many of any kind, go together."""
    s = S.StateVector(n, "enc2b")

    def kernels(gates):
        c = C.Circuit(n)
        for g in gates:
            c.add(*g)
        p = s.plan(c, "pergate")
        names = [k for k, _ in p.launch_info()]
        p.free()
        return names

    h = n - 1
    assert "k_enc_run_in" not in kernels([("CX", h, 0), ("CX", h, 3)])
    assert "k_enc_run_in" not in kernels([("CZ", 0, h), ("CZ", 1, h)])
    if n <= 25:
        assert "k_enc_run_in" not in kernels([("X", 0), ("X", h)])
    assert kernels([("H", 0), ("SX", 3), ("H", h)]) == ["k_enc_run_in"]
    assert kernels([("X", k % 8) for k in range(24)] + [("Z", k % 8) for k in range(24)]) == ["k_enc_run_in"]
