"""Circuits of single-target gates on small registers in one cluster (run_one_launch with
every SM): states and energies against the FP64 oracle for every size of the path, both
types, controls of either value before and after runs, SWAPs, observables of many terms,
circuits too long for the path and gates it does not take."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def circuit(n, seed, length):
    rs = W.rng(seed)
    names = ["H", "X", "Y", "Z", "S", "T", "RX", "RY", "RZ", "SHIFT", "PHASE", "MATRIX", "SWAP"]
    gates = []
    for i in range(length):
        q = [int(v) for v in rs.permutation(n)]
        name = names[rs.integers(len(names))]
        k = 2 if name == "SWAP" else 1
        if n < k:
            continue
        nc = 0 if k == 2 or rs.random() < 0.5 else int(rs.integers(0, min(3, n - k) + 1))
        gates.append(W.Gate(name if nc < 1 or rs.random() < 0.5 else "X", tuple(q[:k]), tuple(q[k:k + nc]),
                            tuple(int(v) for v in rs.integers(0, 2, nc)), theta=float(rs.uniform(-3, 3)),
                            matrix=W.haar_su2(seed + i) if name == "MATRIX" else None))
    return gates


@pytest.mark.parametrize("dt", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("n", [1, 2, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14])
def test_small_circuits_in_one_cluster(dt, n):
    from paper_1912_10877_gb300 import qsim
    tol = 1e-12 if dt == torch.complex128 else 1e-6
    for length in (0, 4, 120, 1500):
        gates = circuit(n, 7 * n + length, length)
        rs = W.rng(n)
        terms = [(float(rs.standard_normal()), tuple((int(q), "Z") for q in rs.permutation(n)[: rs.integers(0, n + 1)]))
                 for _ in range(60)]
        psi = W.haar_state(n, seed=n)
        if dt == torch.complex64:
            psi = psi.astype(np.complex64).astype(np.complex128)
        st = qsim.State(n, dtype=dt).upload(psi)
        circ = qsim.Circuit(gates, n)
        for _ in range(2):  # the second call reuses the circuit's ops
            st.upload(psi)
            out = qsim.run_one_launch(st, circ, None, obs=qsim.Observable(terms))
            st.sync()
        want = oracle.apply_circuit(psi, n, gates)
        assert np.max(np.abs(st.numpy() - want)) < tol, length
        assert abs(float(out.item()) - oracle.expect(want, n, terms)) < 10 * tol, length


def test_parameters_are_read_at_every_call():
    from paper_1912_10877_gb300 import qsim
    n = 9
    gates, _ = W.variational(n, 4, "ring")
    circ, obs = qsim.Circuit(gates, n), qsim.Observable(W.zz_chain(n))
    st = qsim.State(n, dtype=torch.complex128)
    for seed in (1, 2, 1):
        params = W.uniform_angles(circ.nparams, seed)
        st.reset()
        out = qsim.run_one_launch(st, circ, params, obs=obs)
        st.sync()
        want = oracle.apply_circuit(oracle.zero_state(n), n, gates, params)
        assert np.max(np.abs(st.numpy() - want)) < 1e-12
        assert abs(float(out.item()) - oracle.expect(want, n, W.zz_chain(n))) < 1e-12


def test_gates_wider_than_a_block_stay_refused():
    from paper_1912_10877_gb300 import QsimError, qsim
    st = qsim.State(8, dtype=torch.complex128)
    st.reset()
    wide = W.Gate("X", (0,), (1, 2, 3, 4, 5), (1,) * 5)
    with pytest.raises(QsimError):
        qsim.run_one_launch(st, qsim.Circuit([wide], 8), None)


@pytest.mark.parametrize("with_obs", [False, True])
@pytest.mark.parametrize("dt", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("n", [6, 7, 8, 9, 10, 11, 12, 13, 14])
def test_swaps_with_no_barrier_among_the_gates(dt, n, with_obs):
    """Qubits that end elsewhere than they began, with no op that needs a barrier: SWAPs alone
    (exact, many in a row), then with a diagonal gate and gates on lane bits."""
    from paper_1912_10877_gb300 import qsim
    far = [W.Gate("SWAP", (0, n - 1))]
    turn = [W.Gate("SWAP", (q, q + 1)) for q in range(n - 1)]
    mixed = [W.Gate("T", (n - 1,)), W.Gate("H", (0,)), W.Gate("RX", (4,), (n - 1,), (1,), theta=0.3)]
    terms = [(0.5, ((0, "Z"),)), (-1.25, ((n - 1, "Z"), (1, "Z")))] if with_obs else []
    obs = qsim.Observable(terms) if with_obs else None
    st = qsim.State(n, dtype=dt)
    psi = st.upload(W.haar_state(n, seed=n)).numpy().astype(np.complex128)
    tol = 1e-12 if dt == torch.complex128 else 1e-6  # of the path, as above
    for swaps in (far, turn):
        for gates, repeats in ((swaps, 101), (mixed + swaps, 3)):
            st.upload(psi)
            circ, want = qsim.Circuit(gates, n), psi
            for _ in range(repeats):
                out = qsim.run_one_launch(st, circ, None, obs=obs)
                want = oracle.apply_circuit(want, n, gates)
            st.sync()
            if gates is swaps:
                assert np.array_equal(st.numpy().astype(np.complex128), want)
            else:
                assert np.max(np.abs(st.numpy() - want)) < repeats * tol
            if with_obs:
                assert abs(float(out.item()) - oracle.expect(want, n, terms)) < 10 * repeats * tol


@pytest.mark.parametrize("dt", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("n,kmax", [(5, 5), (8, 5), (11, 5), (14, 5), (14, 4), (10, 2)])
def test_gates_piled_on_few_qubits_run_as_blocks(dt, n, kmax):
    """Hundreds of gates on kmax qubits are one block: the same bits as the block launch that the
    caller asks for by its CTAs.  A variational circuit keeps to the cluster (its bits differ)."""
    from paper_1912_10877_gb300 import qsim
    rs = W.rng(n)
    piled = []
    for _ in range(300):
        a, b = (int(v) for v in rs.permutation(kmax)[:2])
        piled.append(W.Gate("RX", (a,), (b,), (1,), theta=float(rs.uniform(-3, 3))))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    psi = W.haar_state(n, seed=n)
    gates, params = W.variational(n, 4, "ring")
    angles = [W.Gate(g.name, g.locs, g.ctrl_locs, g.ctrl_vals, theta=None if g.param is None else float(params[g.param]))
              for g in gates]
    for g, blocks in ((piled, True), (angles, False)):
        if not blocks and (n == 5 or n == 14):
            continue  # near the line between the two
        circ, got = qsim.Circuit(g, n), []
        for ctas in (0, sms):
            st = qsim.State(n, dtype=dt).upload(psi)
            qsim.run_one_launch(st, circ, None, kmax=kmax, grid_ctas=ctas)
            st.sync()
            got.append(st.numpy())
        assert np.array_equal(*got) == blocks
        want = oracle.apply_circuit(psi, n, g)
        assert np.max(np.abs(got[0] - want)) < (1e-12 if dt == torch.complex128 else 2e-5)
