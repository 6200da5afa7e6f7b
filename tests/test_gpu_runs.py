"""Fused runs of the batched and tile engines against the FP64 oracle: runs of uncontrolled
gates on one qubit (rotations, shifts, phases, fixed gates and matrices, up to and beyond
a fused run's length), with controlled X gates before, after and between them (control in
the phase of either value, outside it, two controls), shared parameters, and phases whose
runs leave no room for their sums.  Bounds of tests/test_gpu_batch.py's small batches."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def random_runs(n, seed, length, share=False):
    rs = W.rng(seed)
    gates, p = [], 0
    for _ in range(length):
        t = int(rs.integers(n))
        for _ in range(int(rs.integers(1, 6))):
            kind = rs.integers(9)
            if kind < 6:
                name = ("RX", "RY", "RZ", "RZ", "SHIFT", "PHASE")[kind]
                gates.append(W.Gate(name, (t,), param=p // 2 if share else p))
                p += 1
            elif kind == 6:
                gates.append(W.Gate("MATRIX", (t,), matrix=W.haar_su2(seed + len(gates))))
            else:
                gates.append(W.Gate(("H", "T", "S", "X", "Z", "Y")[rs.integers(6)], (t,)))
        for _ in range(int(rs.integers(0, 3))):
            q = [int(v) for v in rs.permutation(n)]
            target, nc = (t, int(rs.integers(1, 3))) if rs.random() < 0.7 else (q[0], 1)
            ctrl = [v for v in q if v != target][:nc]
            name = "X" if rs.random() < 0.8 else "Z"
            gates.append(W.Gate(name, (target,), tuple(ctrl), tuple(int(v) for v in (rs.random(nc) < 0.8))))
    np_ = (p + 1) // 2 if share else p
    return gates, W.uniform_angles(np_, seed)


@pytest.mark.parametrize("precise,phase", [(False, 4), (False, 3), (False, 2), (True, 3), (True, 2)])
@pytest.mark.parametrize("share", [False, True])
def test_batched_runs(precise, phase, share):
    from paper_1912_10877_gb300 import qsim
    counts = [6, 9, 11, 13, 14]
    specs = [random_runs(n, 17 * n + phase, 40, share) for n in counts]
    obs = [W.zz_chain(n) for n in counts]
    prog = qsim.BatchProgram([qsim.Circuit(g, n, len(p)) for n, (g, p) in zip(counts, specs)],
                             [qsim.Observable(o) for o in obs], phase_qubits=phase, precise=precise)
    st = qsim.State(counts, dtype=torch.complex64)
    params = torch.tensor(np.concatenate([p for _, p in specs]), device="cuda")
    loss, grad = (v.cpu().numpy() for v in prog.run(st, params, grad=True))
    out, off = st.numpy(), 0
    for r, (n, (gates, p)) in enumerate(zip(counts, specs)):
        psi = oracle.apply_circuit(oracle.zero_state(n), n, gates, p)
        wl, wg = oracle.gradient(oracle.zero_state(n), n, gates, p, obs[r])
        assert np.max(np.abs(out[int(st.offsets[r]):int(st.offsets[r + 1])] - psi)) < 2e-5, (r, "state")
        assert abs(loss[r] - wl) < 1e-5, (r, "loss")
        err = np.max(np.abs(grad[off:off + len(p)] - wg))
        assert err < (2e-6 if precise else 1e-5) * max(1.0, np.max(np.abs(wg))), (r, "grad", err)
        off += len(p)


@pytest.mark.parametrize("n,tile", [(9, 9), (12, 10), (15, 13)])
def test_tiled_runs(n, tile):
    from paper_1912_10877_gb300 import qsim
    gates, p = random_runs(n, n, 60)
    terms = W.tfim(n)
    circ = qsim.Circuit(gates, n, len(p))
    st = qsim.State(n, dtype=torch.complex64)
    st.reset()
    st.apply_circuit(circ, p, tiles=True, tile_qubits=tile)
    assert np.max(np.abs(st.numpy() - oracle.apply_circuit(oracle.zero_state(n), n, gates, p))) < 2e-5
    loss, grad = qsim.backward_tiled(st, circ, p, qsim.Observable(terms), tile_qubits=tile)
    wl, wg = oracle.gradient(oracle.zero_state(n), n, gates, p, terms)
    assert abs(loss - wl) < 1e-5
    assert np.max(np.abs(grad - wg)) < 1e-5 * max(1.0, np.max(np.abs(wg)))


def test_phase_with_more_sums_than_room():
    # 64 angles on four qubits, each a run of its own with four sums: only some fuse
    from paper_1912_10877_gb300 import qsim
    n = 6
    gates, p = [], 0
    for layer in range(20):
        for q in range(4):
            gates += [W.Gate("RZ", (q,), param=p), W.Gate("H", (q,))]
            p += 1
        gates += [W.Gate("Z", (q + 1,), (q,)) for q in range(3)]
    params = W.uniform_angles(p, 3)
    prog = qsim.BatchProgram([qsim.Circuit(gates, n)], [qsim.Observable(W.zz_chain(n))])
    st = qsim.State([n], dtype=torch.complex64)
    loss, grad = prog.run(st, torch.tensor(params, device="cuda"), grad=True)
    wl, wg = oracle.gradient(oracle.zero_state(n), n, gates, params, W.zz_chain(n))
    assert abs(float(loss[0]) - wl) < 1e-5
    assert np.max(np.abs(grad.cpu().numpy() - wg)) < 1e-5 * max(1.0, np.max(np.abs(wg)))


@pytest.mark.parametrize("precise", [False, True])
def test_registers_of_one_circuit(precise):
    # a circuit's tables are built once and copied for its other registers
    from paper_1912_10877_gb300 import qsim
    sizes = [8, 14, 8, 6, 14, 8]
    specs = {n: random_runs(n, 5 * n, 30) for n in set(sizes)}
    for n in specs:  # controlled diagonal runs and tables too
        specs[n][0].extend(W.qft(n))
    circ = {n: qsim.Circuit(g, n, len(p)) for n, (g, p) in specs.items()}
    obs = {n: qsim.Observable(W.zz_chain(n)) for n in specs}
    prog = qsim.BatchProgram([circ[n] for n in sizes], [obs[n] for n in sizes], precise=precise)
    st = qsim.State(sizes, dtype=torch.complex64)
    params = [W.uniform_angles(len(specs[n][1]), 100 + r) for r, n in enumerate(sizes)]
    loss, grad = (v.cpu().numpy() for v in prog.run(st, torch.tensor(np.concatenate(params), device="cuda"), grad=True))
    off = 0
    for r, n in enumerate(sizes):
        wl, wg = oracle.gradient(oracle.zero_state(n), n, specs[n][0], params[r], W.zz_chain(n))
        assert abs(loss[r] - wl) < 1e-5, r
        assert np.max(np.abs(grad[off:off + len(wg)] - wg)) < 1e-5 * max(1.0, np.max(np.abs(wg))), r
        off += len(wg)


@pytest.mark.parametrize("count", [223, 255, 480, 511, 512, 513])
def test_passes_at_the_edges_of_their_staged_area(count):
    """One pass of gates that are an op and a gradient record each, up to and past the ops (512) and
    records (224) that its area in shared memory holds: batches of both paths and the tiled gradient.
    Tolerance: 3 x 512 gates (forward, psi and lambda back) of FP32 roundings, 6e-8 each, add up to
    3e-6 at random; six times that."""
    from paper_1912_10877_gb300 import qsim
    n = 14
    rs = W.rng(count)
    gates = []
    for k in range(count):  # four qubits at a time: few phases
        a, b = (int(v) for v in rs.permutation(4)[:2])
        base = 4 * (3 * k // count)
        gates.append(W.Gate("RX", (base + a,), (base + b,), (1,), param=k))
    gates = [W.Gate("H", (q,)) for q in range(n)] + gates
    params, terms = W.uniform_angles(count, count), W.zz_chain(n) + [(0.7, ((2, "Z"),))]
    psi = oracle.apply_circuit(oracle.zero_state(n), n, gates, params)
    wl, wg = oracle.gradient(oracle.zero_state(n), n, gates, params, terms)
    circ, obs = qsim.Circuit(gates, n), qsim.Observable(terms)
    for precise in (False, True):
        st = qsim.State([n, n], dtype=torch.complex64)
        prog = qsim.BatchProgram([circ, circ], [obs, obs], precise=precise)
        loss, grad = prog.run(st, torch.tensor(np.tile(params, 2), device="cuda"), grad=True)
        for r in range(2):
            assert np.max(np.abs(st.register(r).cpu().numpy() - psi)) < 2e-5
            assert abs(float(loss[r]) - wl) < 2e-5
            assert np.max(np.abs(grad[r * count:(r + 1) * count].cpu().numpy() - wg)) < 2e-5 * max(1.0, np.max(np.abs(wg)))
    st = qsim.State(n, dtype=torch.complex64)
    st.reset()
    st.apply_circuit(circ, params, tiles=True)
    assert np.max(np.abs(st.numpy() - psi)) < 2e-5
    loss, grad = qsim.backward_tiled(st, circ, params, obs)
    assert abs(loss - wl) < 2e-5
    assert np.max(np.abs(grad - wg)) < 2e-5 * max(1.0, np.max(np.abs(wg)))
