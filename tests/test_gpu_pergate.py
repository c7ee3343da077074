"""GPU parity of the per-gate path, fused blocks and read-out against the CPU
oracle, through the C ABI.  Tolerances (from the stated accuracy bar):
complex128 max |d amp| <= 1e-12; complex64 1 - F <= 1e-5 and
max |d amp| <= 1e-6 * ||psi||."""

import math

import numpy as np
import pytest

from paper_1912_03243_gb300 import circuits as C

pytestmark = pytest.mark.gpu

TOL_C128 = 1e-12
TOL_C64_F = 1e-5
TOL_C64_AMP = 1e-6


@pytest.fixture(scope="module")
def S():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_03243_gb300 import build, sv

    build.build()
    sv.lib()
    return sv


def fidelity(a, b):
    return abs(np.vdot(a, b)) ** 2 / (np.vdot(a, a).real * np.vdot(b, b).real)


def check(dtype, got, ref):
    got = np.asarray(got, dtype=np.complex128)
    if dtype == "c128":
        assert np.max(np.abs(got - ref)) <= TOL_C128
    else:
        nrm = math.sqrt(np.vdot(ref, ref).real)
        assert np.max(np.abs(got - ref)) <= TOL_C64_AMP * nrm
        assert 1 - fidelity(ref, got) <= TOL_C64_F


def random_u(rng, d=2):
    z = rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d))
    q, r = np.linalg.qr(z)
    return q * (np.diag(r) / np.abs(np.diag(r)))


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 3, 7])
def test_every_target_and_control(S, orc, dtype, n):
    """Every (target, control) pair with a dense, a diagonal (u00 = 1) and a
    general diagonal matrix against the oracle's Eq. 1 loops."""
    rng = np.random.default_rng(100 + n)
    psi0 = C.random_state(n, n)
    mats = [random_u(rng), np.diag([1, np.exp(0.3j)]), np.diag([np.exp(-0.2j), np.exp(0.7j)]),
            orc.gate_matrix("X")]
    sv_ = S.StateVector(n, dtype)
    for u in mats:
        for t in range(n):
            for c in [-1] + [q for q in range(n) if q != t]:
                sv_.from_numpy(psi0)
                sv_.apply_gate(t, u, control=c)
                if c < 0:
                    ref = orc.apply_1q(psi0, t, u)
                else:
                    cu = np.eye(4, dtype=complex)
                    cu[np.ix_([1, 3], [1, 3])] = u
                    ref = orc.apply_kq(psi0, [c, t], cu)
                check(dtype, sv_.to_numpy(), ref)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 5, 11])
def test_matrix_forms(S, orc, dtype, n):
    """Every form the per-gate kernels pick from a matrix's exact entries (real,
    Hadamard, the square roots of X and Y and their adjoints, X, sign flip,
    quarter turns, scaled and signed neighbours of them that must not be taken
    for one), with and without a control, against the oracle's Eq. 1 loops."""
    psi0 = C.random_state(n, 40 + n)
    mats = [orc.gate_matrix(k) for k in ("H", "SX", "SXDG", "SY", "SYDG", "X", "Y", "Z", "S", "SDG", "T")]
    th = 0.4
    mats += [np.array([[np.cos(th), -np.sin(th)], [np.sin(th), np.cos(th)]]), -orc.gate_matrix("H"),
             1j * orc.gate_matrix("SX"), orc.gate_matrix("SY").T, np.diag([1, 1]), np.diag([1j, 1j])]
    sv_ = S.StateVector(n, dtype)
    for u in mats:
        for t, c in {(0, -1), (n - 1, -1), (n // 2, -1), (0, n - 1), (n - 1, 0), (n // 2, 0)}:
            if c == t:
                continue
            sv_.from_numpy(psi0)
            sv_.apply_gate(t, u, control=c)
            if c < 0:
                ref = orc.apply_1q(psi0, t, u)
            else:
                cu = np.eye(4, dtype=complex)
                cu[np.ix_([1, 3], [1, 3])] = u
                ref = orc.apply_kq(psi0, [c, t], cu)
            check(dtype, sv_.to_numpy(), ref)


@pytest.mark.parametrize("dtype,n", [(d, n) for d, top in (("c64", 15), ("c128", 11)) for n in (1, 2, 3, 5, 8, 10, 11, 12, 14, 15)
                                     if n <= top])
def test_small_states_run(S, orc, dtype, n):
    """Plans of small states run many gates per launch (stages of gates on one to
    three target qubits, several launches for long circuits): mixed circuits,
    a QFT, and a run of diagonal gates alone, direct and as a graph replay,
    against the oracle; one launch per gate (sv_plan_execute_timed) agrees."""
    import torch

    diag = C.Circuit(n)
    for q in range(n):
        diag.add("T", q)
        diag.add("CZ" if q else "S", *((q, q - 1) if q else (q,)))
    for c in (C.random_unitary_gates(n, 450 if n >= 5 else 60, n), C.random_circuit(n, 12, 3), C.qft_circuit(n, 1), diag):
        psi0 = C.random_state(n, 70 + n)
        ref = orc.run(c, psi=psi0)
        s = S.StateVector(n, dtype)
        p = s.plan(c, "pergate")
        for _ in range(3):  # direct, capture, replay
            s.from_numpy(psi0)
            p.execute()
            check(dtype, s.to_numpy(), ref)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(p.passes + 1)]
        for e in ev:
            e.record(s.stream)
        s.from_numpy(psi0)
        p.execute_timed(ev)
        check(dtype, s.to_numpy(), ref)
        p.free()


@pytest.mark.parametrize("dtype,n", [("c64", 15), ("c64", 18), ("c64", 23), ("c64", 24), ("c128", 11), ("c128", 12), ("c128", 17),
                                     ("c128", 22), ("c128", 23)])
def test_runs_of_gates(S, orc, dtype, n):
    """Plans of states that stay in L2 run several gates per launch, from the
    smallest to the largest such state and one qubit beyond: mixed circuits
    (controlled and dense gates among them), the random family (complex128 owes
    its scalar factors), a QFT and diagonal gates alone, direct and as a graph
    replay, against the oracle."""
    diag = C.Circuit(n)
    for q in range(n):
        diag.add("T", q)
        diag.add("CZ" if q else "S", *((q, q - 1) if q else (q,)))
    full = [C.random_unitary_gates(n, 300, n), C.random_circuit(n, 12, 3), C.qft_circuit(n, 1), diag]
    for c in full if n <= 18 else [C.random_unitary_gates(n, 60, n), C.random_circuit(n, 3, 3)]:
        psi0 = C.random_state(n, 90 + n)
        ref = orc.run(c, psi=psi0)
        s = S.StateVector(n, dtype)
        p = s.plan(c, "pergate")
        for _ in range(3):  # direct, capture, replay
            s.from_numpy(psi0)
            p.execute()
            check(dtype, s.to_numpy(), ref)
        p.free()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_random_circuit_20q(S, orc, dtype, seed):
    """20 qubits, depth 20 random circuit, full 16 MB vector against the oracle."""
    c = C.random_circuit(20, 20, seed)
    ref = orc.run(c)
    sv_ = S.StateVector(20, dtype)
    sv_.run(c, "pergate")
    check(dtype, sv_.to_numpy(), ref)
    assert abs(sv_.norm() - 1) < (1e-12 if dtype == "c128" else 1e-5)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_all_gate_kinds(S, orc, dtype):
    n = 9
    c = C.random_unitary_gates(n, 300, 17)
    ref = orc.run(c)
    sv_ = S.StateVector(n, dtype)
    sv_.run(c, "pergate")
    check(dtype, sv_.to_numpy(), ref)


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6])
def test_fused_block(S, orc, dtype, k):
    n = 10
    rng = np.random.default_rng(k)
    psi0 = C.random_state(n, 50 + k)
    sv_ = S.StateVector(n, dtype)
    for trial in range(3):
        qs = [int(q) for q in rng.choice(n, size=k, replace=False)]
        u = random_u(rng, 1 << k)
        sv_.from_numpy(psi0)
        sv_.apply_fused(qs, u)
        check(dtype, sv_.to_numpy(), orc.apply_kq(psi0, qs, u))


def test_closed_forms_large(S):
    """GHZ (Sec. 3) and the uniform state at 26 qubits, read out by sampled
    amplitudes and the norm (closed forms, no oracle vector needed)."""
    n = 26
    g = S.StateVector(n, "c64")
    g.run(C.ghz_circuit(n))
    a = g.amplitudes([0, (1 << n) - 1, 1, 12345, 1 << (n - 1)])
    assert np.allclose(a[:2], 1 / math.sqrt(2), atol=1e-7) and np.all(a[2:] == 0)
    assert abs(g.norm() - 1) < 1e-6
    u = S.StateVector(n, "c128")
    u.run(C.uniform_circuit(n))
    idx = np.random.default_rng(0).integers(0, 1 << n, size=1000, dtype=np.uint64)
    assert np.allclose(u.amplitudes(idx), 2.0 ** (-n / 2), rtol=1e-13, atol=0)
    assert abs(u.norm() - 1) < 1e-12


def test_qft_sampled_32q(S):
    """QFT of a basis state at 32 qubits (32 GB, complex64), sampled against
    the closed form 2^{-n/2} exp(2 pi i x y / 2^n)."""
    import torch

    n = 32
    if torch.cuda.mem_get_info()[0] < (8 << n) + (4 << 30):
        pytest.skip("not enough device memory")
    x = 0x9E3779B9
    s = S.StateVector(n, "c64")
    s.set_basis(x)
    s.run(C.qft_circuit(n), "pergate")
    y = np.random.default_rng(1).integers(0, 1 << n, size=4096, dtype=np.uint64)
    got = s.amplitudes(y)
    ph = ((x * y.astype(object)) % (1 << n)).astype(np.float64) / (1 << n)
    expect = np.exp(2j * np.pi * ph) / math.sqrt(1 << n)
    assert np.max(np.abs(got - expect)) <= TOL_C64_AMP
    assert abs(s.norm() - 1) < 1e-4
    del s
    torch.cuda.empty_cache()


@pytest.mark.parametrize("dtype", ["c64", "c128"])
def test_30q_inverse_and_24q_oracle(S, orc, dtype):
    """30 qubits, depth 16: the circuit followed by its inverse returns to
    |0...0>; the same rule at 24 qubits is compared with the oracle."""
    import torch

    c24 = C.random_circuit(24, 16, 1)
    ref = orc.run(c24)
    s24 = S.StateVector(24, dtype)
    s24.run(c24, "pergate")
    check(dtype, s24.to_numpy(), ref)
    del s24
    n = 30
    s = S.StateVector(n, dtype)
    c = C.random_circuit(n, 16, 1)
    s.run(c, "pergate")
    nrm = s.norm()
    s.run(C.inverse_circuit(c), "pergate")
    a = s.amplitudes([0, 1, 2, (1 << n) - 1, 987654321])
    tol = 1e-11 if dtype == "c128" else 2e-5
    assert abs(a[0] - 1) < tol and np.max(np.abs(a[1:])) < tol
    assert abs(nrm - 1) < (1e-12 if dtype == "c128" else 1e-5)
    del s
    torch.cuda.empty_cache()


def test_argument_errors(S):
    s = S.StateVector(5, "c64")
    with pytest.raises(S.SVError) as e:
        s.apply_gate(5, np.eye(2))
    assert e.value.status == 1
    with pytest.raises(S.SVError):
        s.apply_gate(2, np.eye(2), control=2)
    with pytest.raises(S.SVError):
        s.apply_fused([1, 1], np.eye(4))
    with pytest.raises(S.SVError):
        s.amplitudes([32])
    with pytest.raises(S.SVError) as e:
        s.run("qubits 5\nFOO 1\n")
    assert e.value.status == 7
    with pytest.raises(S.SVError):
        s.run("qubits 4\nH 1\n")
    # the state is unchanged by rejected calls
    a = s.amplitudes([0])
    assert a[0] == 1


def test_basis_and_norm(S):
    for dtype in ("c64", "c128", "enc2b"):
        s = S.StateVector(12, dtype)
        s.set_basis(1234)
        a = s.amplitudes([1234, 0])
        assert a[0] == 1 and a[1] == 0
        assert s.norm() == 1.0


@pytest.mark.parametrize("dtype,n", [("c64", 11), ("c64", 19), ("c128", 9), ("c128", 20)])
def test_hadamard_factors_are_owed(S, dtype, n):
    """Runs of gates owe the factor of the library's H: two layers of it on a
    basis state are additions of whole numbers and one power of two, so the
    basis state comes back exactly (with a multiplication per gate 2 c c is one
    place off 1 in both precisions)."""
    c = C.Circuit(n)
    for _ in range(2):
        for q in range(n):
            c.add("H", q)
    s = S.StateVector(n, dtype)
    p = s.plan(c, "pergate")
    for _ in range(3):  # direct, capture, replay
        s.set_basis(5)
        p.execute()
        got = s.to_numpy()
        assert got[5] == 1 and np.count_nonzero(got) == 1
    p.free()


@pytest.mark.parametrize("dtype,n,e", [("c64", 11, 120), ("c64", 18, 120), ("c64", 18, -100), ("c128", 9, 1008), ("c128", 19, 1008),
                                       ("c128", 19, -900)])
def test_unnormalised_states(S, orc, dtype, n, e):
    """Per-gate plans keep room for states far from norm 1: norm 2^120
    (complex128: 2^1008), where a factor owed over many gates would leave the
    type's range, and the smallest ones.  Powers of two are exact, so the
    results are those of the normalised state times 2^e.  Many gates on few
    qubits, so that runs are long."""
    c = C.Circuit(n)
    rng = np.random.default_rng(n)
    for _ in range(100):
        for q in (0, n - 1):
            c.add(str(rng.choice(["H", "SX", "SY", "SXDG", "SYDG", "T"])), q)
    for q in range(n):
        c.add("H", q)
    psi = C.random_state(n, 33)
    ref = orc.run(c, psi=psi)
    s = S.StateVector(n, dtype)
    p = s.plan(c, "pergate")
    for _ in range(3):  # direct, capture, replay
        s.from_numpy(psi * 2.0**e)
        p.execute()
        check(dtype, s.to_numpy().astype(np.complex128) * 2.0**-e, ref)
    p.free()


@pytest.mark.parametrize("dtype,n", [("c64", 9), ("c64", 16), ("c64", 23), ("c64", 24), ("c128", 8), ("c128", 18), ("c128", 23)])
def test_statistics_describe_the_launch_list(S, dtype, n):
    """A per-gate plan's statistics and timing hook describe its list of one
    entry per gate, at every size, however many gates its launches take: the
    entries' bytes add up to the plan's and are those of the gates planned
    alone, and the hook wants one event more than entries."""
    import torch

    c = C.random_circuit(n, 2, 5)
    s = S.StateVector(n, dtype)
    p = s.plan(c, "pergate")
    info = p.launch_info()
    assert p.passes == p.gates == len(info) == len(c)
    assert sum(b for _, b in info) == pytest.approx(p.bytes, rel=1e-12)
    for k in (0, len(c) - 1):
        one = C.Circuit(n)
        one.gates = [c.gates[k]]
        q = s.plan(one, "pergate")
        assert q.launch_info() == [info[k]]
        q.free()
    with pytest.raises(S.SVError):
        p.execute_timed([torch.cuda.Event(enable_timing=True)])
    p.free()


@pytest.mark.parametrize("dtype,n", [("c64", 11), ("c64", 17), ("c128", 9), ("c128", 18), ("c128", 19)])
def test_runs_of_gates_at_the_borders(S, orc, dtype, n):
    """The smallest states that run several gates per launch over many CTAs,
    and both sides of the size at which a thread takes more qubits."""
    test_runs_of_gates(S, orc, dtype, n)


@pytest.mark.parametrize("n", [18, 21])
def test_runs_on_low_qubits(S, orc, n):
    """Runs whose threads hold several of the lowest qubits move their
    amplitudes in rows through shared memory: every combination of two to four
    of qubits 0..5 with high ones, controls in all places, against the oracle."""
    import itertools

    rng = np.random.default_rng(n)
    psi = C.random_state(n, 12).astype(np.complex64).astype(np.complex128)
    s = S.StateVector(n, "c64")
    for k in (2, 3, 4):
        for low in itertools.combinations(range(6), k):
            if n > 18 and (sum(low) + k) % 4:
                continue
            regs = list(low) + [n - 1, 9][: 4 - k]
            c = C.Circuit(n)
            for q in regs:  # (the first gates choose the run's qubits)
                c.add(str(rng.choice(["H", "SX", "SYDG"])), q)
            for q in regs:
                ctl = int(rng.choice([x for x in range(n) if x != q]))
                c.add("T", q)
                c.add("CX", ctl, q)
                c.add("CP", q, (q + 5) % n, 0.3 + q)
            ref = orc.run(c, psi=psi)
            p = s.plan(c, "pergate")
            s.from_numpy(psi)
            p.execute()
            check("c64", s.to_numpy(), ref)
            p.free()


def test_runs_on_low_qubits_are_coalesced(S):
    """Four H on the lowest qubits of a 23-qubit state take no more than two and
    a half times four on the highest (more than four times when every access
    touched a line of its own)."""
    import torch

    n, us = 23, {}
    s = S.StateVector(n, "c64")
    for name, qs in (("low", range(4)), ("high", range(n - 4, n))):
        c = C.Circuit(n)
        for q in qs:
            c.add("H", q)
        p = s.plan(c, "pergate")
        us[name] = 1e9
        for _ in range(8):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            ev[0].record()
            for _ in range(10):
                p.execute()
            ev[1].record()
            torch.cuda.synchronize()
            us[name] = min(us[name], ev[0].elapsed_time(ev[1]) * 100)
        p.free()
    assert us["low"] <= 2.5 * us["high"], us


@pytest.mark.parametrize("dtype,n", [("c64", 23), ("c128", 19), ("c128", 20), ("c128", 22)])
def test_runs_and_launches_of_their_own(S, orc, dtype, n):
    """Plans in which runs of gates that owe factors alternate with diagonal
    gates that keep their own launches, these first, between and last: the
    factors are paid all the same."""
    c = C.Circuit(n)

    def phases():
        for q in (0, 4, 9, n - 2):
            c.add("CP", q, q + 1, 0.2 + 0.1 * q)
        c.add("CZ", 0, n - 1)

    phases()
    for name in ("SX", "H", "SYDG"):
        for q in (0, 3, n - 1):
            c.add(name, q)
        phases()
    psi0 = C.random_state(n, 90 + n)
    ref = orc.run(c, psi=psi0)
    s = S.StateVector(n, dtype)
    p = s.plan(c, "pergate")
    for _ in range(3):  # direct, capture, replay
        s.from_numpy(psi0)
        p.execute()
        check(dtype, s.to_numpy(), ref)
    p.free()


@pytest.mark.parametrize("dtype,n", [("c64", 23), ("c128", 22), ("c128", 20)])
def test_diagonal_gates_are_not_slower_together(S, dtype, n):
    """Controlled phases on a large state, each of which visits a quarter of it,
    take no longer in one plan than in a plan each (and a fifth)."""
    import torch

    c = C.Circuit(n)
    for q in range(n - 1):
        c.add("CP", q, q + 1, 0.1 + 0.1 * q)
    if dtype == "c64":
        c.gates = c.gates[-2:]
    s = S.StateVector(n, dtype)
    alone = []
    for g in c.gates:
        one = C.Circuit(n)
        one.gates = [g]
        alone.append(s.plan(one, "pergate"))
    us = {}
    for name, plans in (("together", [s.plan(c, "pergate")]), ("alone", alone)):
        us[name] = 1e9
        for _ in range(8):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            ev[0].record()
            for _ in range(10):
                for p in plans:
                    p.execute()
            ev[1].record()
            torch.cuda.synchronize()
            us[name] = min(us[name], ev[0].elapsed_time(ev[1]) * 100)
        for p in plans:
            p.free()
    assert us["together"] <= 1.2 * us["alone"], us
