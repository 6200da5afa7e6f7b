"""Small registers, whose gates run many to a launch inside a thread-block cluster: bit for
bit the amplitudes of the launch-a-gate path (which a batch with more amplitudes takes),
and the FP64 oracle's; every size of the path, targets and controls on lanes, threads,
a thread's amplitudes and other CTAs, lists longer than a launch takes, gates in between
that the path does not take, batches, per-register parameters."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

TDT = {"c64": torch.complex64, "c128": torch.complex128}
TOL = {"c64": 2e-5, "c128": 1e-12}


def random_circuit(n, seed, length):
    rs = W.rng(seed)
    names = ["H", "X", "Y", "Z", "S", "T", "RX", "RY", "RZ", "SHIFT", "PHASE", "MATRIX", "SWAP", "ROT"]
    gates = []
    for i in range(length):
        q = [int(v) for v in rs.permutation(n)]
        name = names[rs.integers(len(names))]
        k = 2 if name in ("SWAP", "ROT") else 1
        if n < k:
            continue
        nc = int(rs.integers(0, min(3, n - k) + 1))
        ctrl, vals = tuple(q[k:k + nc]), tuple(int(v) for v in rs.integers(0, 2, nc))
        gates.append(W.Gate(name, tuple(q[:k]), ctrl, vals, theta=float(rs.uniform(-3, 3)),
                            paulis="XZ" if name == "ROT" and i % 5 == 0 else "ZZ" if name == "ROT" else None,
                            matrix=W.haar_su2(seed + i) if name == "MATRIX" else None))
    return gates


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n", [1, 2, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14])
def test_small_registers(dt, n):
    from paper_1912_10877_gb300 import qsim
    for length in (3, 60, 700):
        gates = random_circuit(n, 31 * n + length, length)
        circ = qsim.Circuit(gates, n)
        psi = W.haar_state(n, seed=n)
        st = qsim.State(n, dtype=TDT[dt]).upload(psi)
        st.apply_circuit(circ)
        got = st.numpy()
        if length < 700 or n < 9:
            assert np.max(np.abs(got - oracle.apply_circuit(psi, n, gates))) < TOL[dt], length
        many = (1 << 17 >> n) + 1  # one register more than the path takes
        if dt == "c64" and n < 10:
            continue               # such a batch runs on the tile engine
        big = qsim.State(n, dtype=TDT[dt], nbatch=many).upload(np.tile(psi, many))
        big.apply_circuit(circ)
        ref = big.register(many - 1).cpu().numpy()
        assert np.array_equal(got, ref), (length, np.max(np.abs(got - ref)))


@pytest.mark.parametrize("dt", ["c64", "c128"])
def test_small_batches_and_per_register_parameters(dt):
    from paper_1912_10877_gb300 import qsim
    n, nreg = 9, 5
    gates, _ = W.variational(n, 3, "ring")
    params = np.stack([W.uniform_angles(27 * n // 3, 50 + r) for r in range(nreg)])
    circ = qsim.Circuit(gates, n)
    psi = [W.haar_state(n, seed=r) for r in range(nreg)]
    st = qsim.State(n, dtype=TDT[dt], nbatch=nreg).upload(np.concatenate(psi))
    st.apply_circuit(circ, params, per_register=True)
    out = st.numpy().reshape(nreg, -1)
    for r in range(nreg):
        assert np.max(np.abs(out[r] - oracle.apply_circuit(psi[r], n, gates, params[r]))) < TOL[dt]
    st.upload(np.concatenate(psi))
    st.apply_circuit(circ, params[0])
    out = st.numpy().reshape(nreg, -1)
    for r in range(nreg):
        assert np.max(np.abs(out[r] - oracle.apply_circuit(psi[r], n, gates, params[0]))) < TOL[dt]


@pytest.mark.parametrize("dt", ["c64", "c128"])
def test_short_lists_and_dense_layers_keep_their_bits(dt):
    """Lists that go gate by gate (one gate; at 14 qubits complex128 dense gates alone) and their
    neighbours that do not: the bits of a launch a gate in the same order."""
    from paper_1912_10877_gb300 import qsim
    for n in (1, 3, 10, 13, 14):
        psi = W.haar_state(n, seed=n)
        layer = [W.Gate("MATRIX", (q,), matrix=W.haar_su2(q)) for q in range(n)]
        real = [W.Gate("H", (q,)) for q in range(n)]
        for gates in (layer[:1], real[:1], layer, real, [W.Gate("T", (0,), (n - 1,))] + layer if n > 1 else real):
            circ, got = qsim.Circuit(gates, n), []
            for fused in (True, False):
                got.append(qsim.State(n, dtype=TDT[dt]).upload(psi).apply_circuit(circ, fused=fused).numpy())
            assert np.array_equal(*got), (n, len(gates))
