"""The tile engine's runs of diagonal gates and its swap passes against the FP64 oracle
(2e-5 absolute, the engine's tolerance): runs whose entries lie on lane, warp and
tile-id bits and on several of them, scalar entries, factors other than 1 on both
values; swap networks before and after the passes, on odd and even sizes, on the rows'
own qubits, whole and partial; and the gradient through them."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def apply_tiles(n, gates, tile, nbatch=1, params=None):
    from paper_1912_10877_gb300 import qsim
    psi = [W.haar_state(n, seed=n + r) for r in range(nbatch)]
    st = qsim.State(n, dtype=torch.complex64, nbatch=nbatch)
    st.upload(np.concatenate(psi))
    st.apply_circuit(qsim.Circuit(gates, n), params, tiles=True, tile_qubits=tile)
    out = st.numpy().reshape(nbatch, -1)
    for r in range(nbatch):
        assert np.max(np.abs(out[r] - oracle.apply_circuit(psi[r], n, gates, params))) < 2e-5, (n, tile, r)


def diagonal_runs(n, seed):
    rs = W.rng(seed)
    gates = []
    for t in rs.permutation(n):
        gates.append(W.Gate("H", (int(t),)))
        for _ in range(12):
            q = [int(x) for x in rs.permutation(n) if x != t][: rs.integers(1, 3)]
            name = ("SHIFT", "RZ", "PHASE", "T", "Z", "SDG")[rs.integers(6)]
            gates.append(W.Gate(name, (int(t),), tuple(q), tuple(int(v) for v in rs.integers(0, 2, len(q))),
                                theta=float(rs.uniform(-3, 3))))
        for _ in range(4):
            gates.append(W.Gate(("RZ", "SHIFT", "S")[rs.integers(3)], (int(rs.integers(n)),), theta=float(rs.uniform(-3, 3))))
    return gates


@pytest.mark.parametrize("n,tile", [(9, 9), (11, 9), (13, 13), (16, 10), (17, 13)])
def test_runs_of_diagonal_gates(n, tile):
    apply_tiles(n, diagonal_runs(n, n), tile)


def layers(n, seed):
    """A real gate on a qubit, then phases on it: inside the phase, outside, both, with
    controls of either value, and now and then a gate that acts on the 0 as well."""
    rs = W.rng(seed)
    gates = []
    for t in rs.permutation(n):
        t = int(t)
        gates.append(W.Gate("H", (t,)) if rs.integers(2) else W.Gate("RY", (t,), theta=float(rs.uniform(-3, 3))))
        for q in rs.permutation(n)[: rs.integers(2, n)]:
            if q == t:
                continue
            a, b = (t, int(q)) if rs.integers(4) else (int(q), t)
            gates.append(W.Gate(("SHIFT", "T", "Z", "S")[rs.integers(4)], (a,), (b,), (int(rs.integers(8) > 0),),
                                theta=float(rs.uniform(-3, 3))))
        if rs.integers(6) == 0:
            gates.append(W.Gate("RZ", (t,), (int((t + 1) % n),), (1,), theta=0.4))
    return gates


@pytest.mark.parametrize("n,tile", [(9, 9), (11, 9), (13, 13), (16, 10), (18, 13)])
def test_real_gates_with_their_phases(n, tile):
    for seed in (1, 2):
        apply_tiles(n, layers(n, 10 * n + seed), tile)
    qft = [g for t in reversed(range(n)) for g in
           [W.Gate("H", (t,))] + [W.Gate("SHIFT", (t,), (c,), (1,), theta=np.pi / 2 ** (t - c)) for c in range(t)]]
    apply_tiles(n, qft, tile, 2)


@pytest.mark.parametrize("reps", [3, 6, 12, 40])
def test_passes_that_outgrow_shared_memory(reps):
    """One pass of more and more phases, ops, runs and tables than its staged area holds."""
    n = 11
    apply_tiles(n, [g for k in range(reps) for g in layers(n, 100 + k)], 13)


def networks(n):
    rs = W.rng(n)
    half = n // 2
    yield [(i, n - 1 - i) for i in range(half)]
    yield [(0, 1), (2, 3)]
    yield [(4, 5), (1, n - 1)]
    yield [tuple(int(q) for q in pair) for pair in rs.permutation(n)[: 2 * half].reshape(-1, 2)]


@pytest.mark.parametrize("n,tile,nbatch", [(16, 13, 1), (17, 11, 2), (19, 13, 1), (20, 9, 1)])
def test_swap_networks(n, tile, nbatch):
    for net in networks(n):
        swaps = [W.Gate("SWAP", p) for p in net]
        core = [W.Gate("RY", (q,), theta=0.3 + q) for q in (0, n // 2)] + [W.cnot(1, n - 2)]
        for gates in (swaps, core + swaps, swaps + core, swaps + core + swaps[::-1], core + swaps + swaps[:1]):
            apply_tiles(n, gates, tile, nbatch)


def test_gradient_through_swap_networks():
    from paper_1912_10877_gb300 import qsim
    n = 16
    swaps = [W.Gate("SWAP", (i, n - 1 - i)) for i in range(n // 2)]
    core, params = W.variational(n, 2, "ring", seed=3)
    gates = swaps + core + swaps
    terms = [(1.0, ((0, "Z"), (3, "Z"))), (0.5, ((n - 1, "X"),))]
    st = qsim.State(n, dtype=torch.complex64)
    st.reset()
    circ = qsim.Circuit(gates, n)
    st.apply_circuit(circ, params, tiles=True, tile_qubits=9)
    loss, grad = qsim.backward_tiled(st, circ, params, qsim.Observable(terms), tile_qubits=9)
    wl, wg = oracle.gradient(oracle.zero_state(n), n, gates, params, terms)
    assert abs(loss - wl) < 1e-5
    assert np.max(np.abs(grad - wg)) < 1e-5 * np.max(np.abs(wg))  # the tiled gradient's bound is 3e-6 at n = 22


@pytest.mark.parametrize("n", [16, 21])
def test_swap_passes_keep_the_schedule(n):
    from paper_1912_10877_gb300 import qsim
    circ = qsim.Circuit(W.qft(n, swaps=True), n)
    order, passes = qsim.tile_order(circ, 0)
    assert sorted(order.tolist()) == list(range(n * (n + 1) // 2 + 3 * (n // 2)))
    assert qsim.schedule_info(circ)[0] == passes[-1] + 1
