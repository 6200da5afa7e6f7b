"""The FP64 backward walk's fused runs against the oracle: random circuits of runs on one
qubit (longer than a pass takes, diagonal ones, with matrices and fixed gates), controlled
X gates before, after and between them, shared parameters, checkpoints that cut runs, on
one qubit and up.  complex128: 1e-11 of the largest gradient entry (FP64 sums of up to
2^13 products of unit-norm states through a few hundred gates); complex64 with
checkpoints: 1e-5, the storage rounding of its states."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def circuit(n, seed, length):
    rs = W.rng(seed)
    gates, p = [], 0
    for _ in range(length):
        t = int(rs.integers(n))
        for _ in range(int(rs.integers(1, 12))):
            kind = rs.integers(10)
            if kind < 7:
                name = ("RX", "RY", "RZ", "RZ", "SHIFT", "PHASE", "ROT")[kind]
                gates.append(W.Gate(name, (t,), param=p if rs.random() < 0.9 or not p else p - 1,
                                    paulis="XYZ"[rs.integers(3)] if name == "ROT" else None))
                p = max(p, gates[-1].param + 1)
            elif kind == 7:
                gates.append(W.Gate("MATRIX", (t,), matrix=W.haar_su2(seed + len(gates))))
            else:
                gates.append(W.Gate(("H", "T", "S", "X", "Z", "Y")[rs.integers(6)], (t,)))
        for _ in range(int(rs.integers(0, 3)) if n > 1 else 0):
            q = [int(v) for v in rs.permutation(n)]
            target = t if rs.random() < 0.7 else q[0]
            ctrl = [v for v in q if v != target][: int(rs.integers(1, 3))]
            vals = tuple(int(v) for v in (rs.random(len(ctrl)) < 0.7))
            gates.append(W.Gate("X" if rs.random() < 0.8 else "RY", (target,), tuple(ctrl), vals, theta=0.4))
        if n > 2 and rs.random() < 0.2:
            q = [int(v) for v in rs.permutation(n)[:2]]
            gates.append(W.Gate("ROT", tuple(q), param=p, paulis="XY"))
            p += 1
    return gates, W.uniform_angles(p, seed)


@pytest.mark.parametrize("n", [1, 2, 5, 9, 10, 13])
@pytest.mark.parametrize("every", [0, 7, 50])
def test_gradient_of_runs(n, every):
    from paper_1912_10877_gb300 import qsim
    gates, params = circuit(n, 10 * n + every, 30)
    terms = W.tfim(n)
    circ, obs = qsim.Circuit(gates, n, len(params)), qsim.Observable(terms)
    wl, wg = oracle.gradient(oracle.zero_state(n), n, gates, params, terms)
    for dtype, tol in ((torch.complex128, 1e-11), (torch.complex64, 1e-5)):
        st = qsim.State(n, dtype=dtype)
        st.reset()
        ck = qsim.checkpoint_buffer(st, circ, every)
        if every:
            qsim.apply_circuit_ckpt(st, circ, params, every, ck)
        else:
            st.apply_circuit(circ, params)
        loss, grad = qsim.backward(st, circ, params, obs, every if ck is not None else 0, ck)
        scale = max(1.0, np.max(np.abs(wg)))
        assert abs(loss - wl) < tol * max(1.0, abs(wl))
        assert np.max(np.abs(grad - wg)) < tol * scale, (dtype, np.max(np.abs(grad - wg)) / scale)


@pytest.mark.parametrize("n,every", [(2, 0), (3, 500), (10, 900)])
def test_gradient_of_many_runs(n, every):
    """Runs whose matrices have entries of one size, more than any factor that psi and
    lambda carry may grow through: the bounds of the short circuits times the gates."""
    from paper_1912_10877_gb300 import qsim
    rs = W.rng(n)
    gates = []
    for k in range(600):
        t = k % n
        gates += [W.Gate("RX", (t,), theta=np.pi / 2 + float(rs.uniform(-0.1, 0.1))), W.Gate("RZ", (t,), param=k)]
        gates.append(W.Gate("X", (t,), ((t + 1) % n,), (k % 3 > 0,)))
    params = W.uniform_angles(600, n)
    terms = W.tfim(n)
    circ, obs = qsim.Circuit(gates, n, len(params)), qsim.Observable(terms)
    wl, wg = oracle.gradient(oracle.zero_state(n), n, gates, params, terms)
    st = qsim.State(n, dtype=torch.complex128)
    st.reset()
    ck = qsim.checkpoint_buffer(st, circ, every)
    if every:
        qsim.apply_circuit_ckpt(st, circ, params, every, ck)
    else:
        st.apply_circuit(circ, params)
    loss, grad = qsim.backward(st, circ, params, obs, every if ck is not None else 0, ck)
    assert abs(loss - wl) < 1e-10 * max(1.0, abs(wl))
    assert np.max(np.abs(grad - wg)) < 1e-10 * max(1.0, np.max(np.abs(wg)))


@pytest.mark.parametrize("n", [2, 5, 9, 13])
def test_compensated_gate_with_an_x_is_the_two_of_them(n):
    from paper_1912_10877_gb300 import qsim
    rs = W.rng(n)
    psi = W.haar_state(n, seed=n)
    gates = []
    for _ in range(40):
        q = [int(v) for v in rs.permutation(n)]
        k = int(rs.integers(1, min(4, n)))
        gates.append(W.Gate(("H", "RX", "RY", "Y", "T", "MATRIX")[rs.integers(6)], (q[0],), theta=float(rs.uniform(-3, 3)),
                            matrix=W.haar_su2(len(gates))))
        gates.append(W.Gate("X", (q[0],), tuple(q[1:1 + k]), tuple(int(v) for v in rs.integers(0, 2, k))))
    fused, apart = qsim.State(n, dtype=torch.complex64), qsim.State(n, dtype=torch.complex64)
    fused.upload(psi)
    apart.upload(psi)
    fused.apply_circuit(qsim.Circuit(gates, n), precise=True)
    for g in gates:
        apart.apply_circuit(qsim.Circuit([g], n), precise=True)
    assert np.array_equal(fused.numpy(), apart.numpy())  # the X only renames
