"""The work this simulator is measured on, through its public entry points.

Every case is one call, or one short sequence of calls, that a user's program
makes: applying a circuit, a training step with the gradient of an energy, an
expectation value and samples, a Hamiltonian's sparse matrix.  The sizes are
those of the repository's workloads (small variational circuit, single-gate
suite, batch of uneven registers, differentiation, large register) and of the
paper's listings (QFT on a random state, mat(heisenberg(20)), shot-based
gradients); `draw` spreads them over the ranges a user would run.

A complex64 register's losses and gradients are returned in float32, the type a
training program keeps its angles in; complex128 ones stay float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads as W
from paper_1912_10877_gb300 import autograd, qsim

DTYPES = {"c64": torch.complex64, "c128": torch.complex128}
SHOTS = 1024


def listed():
    return [
        # the smallest call: the paper's QFT listing on rand_state(10); launches and latency count
        {"name": "qft_n10_c128", "kind": "qft", "n": 10, "dtype": "c128", "swaps": False},
        # a QFT with its swap network on a register far larger than L2 (tile engine)
        {"name": "qft_n29_c64", "kind": "qft", "n": 29, "dtype": "c64", "swaps": True},
        # small variational workload: 10 layers on 12 qubits and <sum ZZ>, one energy evaluation of an optimiser
        {"name": "vqe_n12_c128", "kind": "vqe", "n": 12, "dtype": "c128", "depth": 10, "ring": False},
        # the single-gate suite, an interactive user's gate-by-gate program, both precisions
        {"name": "gates_n25_c64", "kind": "gates", "n": 25, "dtype": "c64"},
        {"name": "gates_n25_c128", "kind": "gates", "n": 25, "dtype": "c128"},
        # a training step of the batched engine: 1024 uneven registers, forward and gradient
        {"name": "batch_1024_c64", "kind": "batch", "nreg": 1024, "lo": 10, "hi": 18, "depth": 20, "precise": False},
        # the same step in the precise mode on a smaller batch, whose largest registers set its length
        {"name": "batch_200_precise", "kind": "batch", "nreg": 200, "lo": 10, "hi": 16, "depth": 20, "precise": True},
        # differentiation workload: energy and gradient of 6000 angles through torch autograd, checkpoints each 10 layers
        {"name": "train_n20_c64", "kind": "train", "n": 20, "depth": 100, "ckpt_layers": 10},
        # random brickwork circuit through fused 5-qubit blocks, forward and reversible gradient (state larger than L2)
        {"name": "brickwork_n26_c64", "kind": "brickwork", "n": 26, "depth": 20},
        # reading a prepared register: the Ising energy and a batch of samples
        {"name": "observe_n25_c64", "kind": "observe", "n": 25, "dtype": "c64", "shots": 4096},
        # mat(heisenberg(20)): the Hamiltonian as a sparse matrix
        {"name": "matrix_n20", "kind": "matrix", "n": 20},
        # shot-based parameter-shift gradient of the Ising energy
        {"name": "shots_n10_c64", "kind": "shots", "n": 10, "dtype": "c64", "depth": 4, "shots": SHOTS},
    ]


def draw(rng):
    kind = rng.choice(["qft", "qft", "vqe", "gates", "batch", "batch", "train", "brickwork", "observe", "matrix", "shots"])
    dtype = rng.choice(["c64", "c64", "c128"])
    if kind == "qft":
        return {"kind": kind, "n": rng.randint(6, 28 if dtype == "c64" else 24), "dtype": dtype,
                "swaps": rng.random() < 0.5}
    if kind == "vqe":
        return {"kind": kind, "n": rng.randint(5, 15), "dtype": dtype, "depth": rng.randint(2, 16),
                "ring": rng.random() < 0.5}
    if kind == "gates":
        return {"kind": kind, "n": rng.randint(14, 27 if dtype == "c64" else 25), "dtype": dtype}
    if kind == "batch":
        lo = rng.randint(6, 11)
        precise = rng.random() < 0.4
        return {"kind": kind, "nreg": int(2 ** rng.uniform(3, 8 if precise else 9.5)), "lo": lo,
                "hi": lo + rng.randint(1, 5 if precise else 7), "depth": rng.randint(4, 20), "precise": precise}
    if kind == "train":
        return {"kind": kind, "n": rng.randint(9, 21), "depth": rng.randint(12, 40), "ckpt_layers": rng.choice([0, 5, 10])}
    if kind == "brickwork":
        return {"kind": kind, "n": rng.randint(18, 26), "depth": rng.randint(4, 20)}
    if kind == "observe":
        return {"kind": kind, "n": rng.randint(14, 27 if dtype == "c64" else 26), "dtype": dtype,
                "shots": int(2 ** rng.uniform(5, 14))}
    if kind == "matrix":
        return {"kind": kind, "n": rng.randint(10, 21)}
    return {"kind": "shots", "n": rng.randint(6, 12), "dtype": dtype, "depth": rng.randint(1, 4),
            "shots": int(2 ** rng.uniform(6, 11))}


# ------------------------------------------------------------------ inputs shared by the calls and their exact values

def _random_amplitudes(n, dtype, seed):
    """A Haar-random state made on the device: normalised complex Gaussians."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(1 << n, dtype=DTYPES[dtype], device="cuda", generator=g)
    return v.div_(torch.linalg.vector_norm(torch.view_as_real(v), dtype=torch.float64))


def _register(n, dtype, seed):
    st = qsim.State(n, dtype=DTYPES[dtype])
    st.buffer.copy_(_random_amplitudes(n, dtype, seed))
    return st


def _angles(count, seed, dtype=np.float64):
    return W.uniform_angles(count, seed).astype(dtype)


def _entangler(case):
    return "ring" if case.get("ring") else "ladder"


def _batch_counts(case):
    return [int(x) for x in W.batch_qubit_counts(case["nreg"], case["lo"], case["hi"], 0)]


def _batch_inputs(case, seed):
    """(register sizes, {size: gate list}, angles per register as float32)."""
    counts = _batch_counts(case)
    gates = {n: W.variational(n, case["depth"], "ladder")[0] for n in sorted(set(counts))}
    angles = [_angles(3 * n * case["depth"], seed + 1 + r, np.float32) for r, n in enumerate(counts)]
    return counts, gates, angles


def _shot_inputs(case, seed):
    gates, params = W.variational(case["n"], case["depth"], "ladder", seed=seed)
    return gates, params, W.rng(seed + 1).random((2, 2 * len(params), case["shots"]))


def prepare(case, seed):
    kind, n = case["kind"], case.get("n")
    s = {"case": case}
    if kind == "qft":
        s["state"] = _register(n, case["dtype"], seed)
        s["circuit"] = qsim.Circuit(W.qft(n, case["swaps"]), n)
    elif kind == "vqe":
        gates, s["params"] = W.variational(n, case["depth"], _entangler(case), seed=seed)
        s["state"] = qsim.State(n, dtype=DTYPES[case["dtype"]])
        s["circuit"], s["obs"] = qsim.Circuit(gates, n), qsim.Observable(W.zz_chain(n))
    elif kind == "gates":
        s["state"] = _register(n, case["dtype"], seed)
        s["gates"] = [g for _, g in W.single_gate_suite(n)]
    elif kind == "batch":
        counts, gates, angles = _batch_inputs(case, seed)
        circuits = {k: qsim.Circuit(g, k) for k, g in gates.items()}
        obs = {k: qsim.Observable(W.zz_chain(k)) for k in gates}
        s["program"] = qsim.BatchProgram([circuits[k] for k in counts], [obs[k] for k in counts], precise=case["precise"])
        s["state"] = qsim.State(counts, dtype=torch.complex64)
        s["params"] = torch.tensor(np.concatenate(angles), device="cuda")
    elif kind == "train":
        gates, _ = W.variational(n, case["depth"], "ring", params=())
        s["circuit"], s["obs"] = qsim.Circuit(gates, n), qsim.Observable(W.tfim(n))
        s["every"] = case["ckpt_layers"] * (len(gates) // case["depth"])
        s["params"] = torch.tensor(_angles(3 * n * case["depth"], seed, np.float32), device="cuda", requires_grad=True)
    elif kind == "brickwork":
        gates, s["params"] = W.brickwork(n, case["depth"], seed=seed)
        s["state"] = qsim.State(n, dtype=torch.complex64)
        s["work"] = torch.empty(8 << n, dtype=torch.uint8, device="cuda")
        s["circuit"], s["obs"] = qsim.Circuit(gates, n), qsim.Observable(W.z_on(0))
    elif kind == "observe":
        s["state"], s["obs"] = _register(n, case["dtype"], seed), qsim.Observable(W.tfim(n))
        s["seed"] = seed
    elif kind == "matrix":
        s["obs"] = qsim.Observable([(c * j, ops) for (c, ops), j in zip(W.heisenberg(n), _couplings(n, seed))])
    else:
        gates, s["params"], s["uniforms"] = _shot_inputs(case, seed)
        s["circuit"], s["obs"] = qsim.Circuit(gates, n), qsim.Observable(W.tfim(n))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "qft":
        s["state"].apply_circuit(s["circuit"])
        return s["state"].tensor()
    if kind == "vqe":
        s["state"].reset()
        energy = qsim.run_one_launch(s["state"], s["circuit"], s["params"], kmax=5, obs=s["obs"])
        return s["state"].tensor(), energy.to(torch.float32) if case["dtype"] == "c64" else energy
    if kind == "gates":
        for g in s["gates"]:
            s["state"].apply(g)
        return s["state"].tensor()
    if kind == "batch":
        loss, grad = s["program"].run(s["state"], s["params"].double(), grad=True)
        return s["state"].buffer, loss.float(), grad.float()
    if kind == "train":
        s["params"].grad = None
        loss = autograd.expectation(s["params"], s["circuit"], s["obs"], torch.complex64, s["every"])
        loss.backward()
        return loss.detach(), s["params"].grad
    if kind == "brickwork":
        s["state"].reset()
        s["state"].apply_circuit(s["circuit"], s["params"], blocks=5)
        loss, grad = qsim.backward_blocks(s["state"], s["circuit"], s["params"], s["obs"], kmax=5, work=s["work"])
        return np.float32(loss), grad.astype(np.float32), s["state"].tensor()
    if kind == "observe":
        return s["state"].expect(s["obs"]), s["state"].measure_seeded(s["seed"], case["shots"])
    if kind == "matrix":
        return qsim.observable_csr(s["obs"], case["n"])
    return qsim.faithful_gradient(s["circuit"], s["params"], s["obs"], dtype=DTYPES[case["dtype"]],
                                  nshots=case["shots"], uniforms=s["uniforms"])


def work(case):
    """Bytes of the inputs and outputs, and the arithmetic of the method in its usual form: a dense
    2x2 gate 14 operations an amplitude, a diagonal factor 6, a Hadamard 4, an Rx 6; a rotation run
    forward, uncomputed on psi and lambda and its three derivatives 64 an amplitude."""
    kind, n = case["kind"], case.get("n", 0)
    dim = 1 << n
    amp = 16 if case.get("dtype") == "c128" else 8
    if kind == "qft":
        return {"bytes": 2 * amp * dim, "flops": dim * (4 * n + 1.5 * n * (n - 1) / 2)}
    if kind == "vqe":
        return {"bytes": amp * dim + 24 * n * case["depth"], "flops": 14 * dim * n * case["depth"]}
    if kind == "gates":
        # amplitudes a gate changes, read and written: all for X, H, Rx; half for T and CNOT; a quarter for Toffoli
        return {"bytes": 2 * amp * dim * (3 * n + n / 2 + 3 / 2 + 2 / 4), "flops": dim * n * (4 + 6 + 3)}
    if kind == "batch":
        counts = _batch_counts(case)
        return {"bytes": sum((8 << k) + 8 * 3 * k * case["depth"] for k in counts),
                "flops": sum(64.0 * k * case["depth"] * (1 << k) for k in counts)}
    if kind == "train":
        return {"bytes": 8 * 3 * n * case["depth"], "flops": 64.0 * n * case["depth"] * dim}
    if kind == "brickwork":
        # forward, and two states uncomputed with one derivative a gate
        return {"bytes": amp * dim + 12 * n * case["depth"], "flops": n * case["depth"] * dim * (3 * 14 + 4)}
    if kind == "observe":
        return {"bytes": 2 * amp * dim + 8 * case["shots"], "flops": dim * (3 + 2 * n + 2 * n)}
    if kind == "matrix":
        # n 2^(n-1) flips of unequal neighbours and a diagonal; a row pointer a row
        return {"bytes": 24 * (n * dim // 2 + dim) + 8 * dim, "flops": 3 * n * dim}
    registers = 2 * 3 * n * case["depth"]
    return {"bytes": 8 * registers * (2 * case["shots"]) + 4 * registers,
            "flops": registers * dim * (14 * n * case["depth"] + 2 * 4)}


# ------------------------------------------------------------------ exact values: plain torch in complex128

def _view(psi, n, qubits):
    """psi [R, 2^n] with an axis of its own for each of `qubits`, highest first."""
    shape, hi = [psi.shape[0]], n
    for q in sorted(qubits, reverse=True):
        shape += [1 << (hi - 1 - q), 2]
        hi = q
    return psi.view(shape + [1 << hi])


def _slice(psi, n, values):
    """The amplitudes whose qubit q holds values[q]."""
    at = [slice(None)]
    for q in sorted(values, reverse=True):
        at += [slice(None), values[q]]
    return _view(psi, n, values)[tuple(at + [slice(None)])]


def _gate(g, theta, dagger=False):
    """Rows of a one-target gate; theta is a number or one number a register."""
    if g.name == "MATRIX":
        m = np.asarray(g.matrix, dtype=complex)
        u = [[complex(m[0, 0]), complex(m[0, 1])], [complex(m[1, 0]), complex(m[1, 1])]]
    elif g.name in ("X", "Z", "H", "T"):
        h = math.sqrt(0.5)
        u = {"X": [[0, 1], [1, 0]], "Z": [[1, 0], [0, -1]], "H": [[h, h], [h, -h]],
             "T": [[1, 0], [0, complex(h, h)]]}[g.name]
    else:
        t = torch.as_tensor(theta, dtype=torch.float64, device="cuda").reshape(-1, 1, 1)
        t = t if t.numel() > 1 else t.cpu().reshape(())
        half = (t / 2).to(torch.complex128)
        e = {"RX": [[torch.cos(half), -1j * torch.sin(half)], [-1j * torch.sin(half), torch.cos(half)]],
             "RZ": [[torch.exp(-1j * half), 0], [0, torch.exp(1j * half)]],
             "SHIFT": [[1, 0], [0, torch.exp(2j * half)]]}[g.name]
        u = [[complex(x) if torch.is_tensor(x) and x.dim() == 0 else x for x in row] for row in e]
    if dagger:
        conj = lambda x: x.conj() if torch.is_tensor(x) else complex(x).conjugate()  # noqa: E731
        u = [[conj(u[0][0]), conj(u[1][0])], [conj(u[0][1]), conj(u[1][1])]]
    return u


def _is(x, value):
    return not torch.is_tensor(x) and x == value


def _apply(psi, n, g, theta=None, dagger=False):
    ctrl = dict(zip(g.ctrl_locs, g.ctrl_vals))
    if g.name == "SWAP":
        i, j = g.locs
        a, b = _slice(psi, n, {i: 0, j: 1}), _slice(psi, n, {i: 1, j: 0})
        t = a.clone()
        a.copy_(b)
        b.copy_(t)
        return
    t = g.locs[0]
    a, b = _slice(psi, n, {**ctrl, t: 0}), _slice(psi, n, {**ctrl, t: 1})
    (u00, u01), (u10, u11) = _gate(g, theta, dagger)
    wide = lambda u: u.view([-1] + [1] * (a.dim() - 1)) if torch.is_tensor(u) else u  # noqa: E731
    u00, u01, u10, u11 = wide(u00), wide(u01), wide(u10), wide(u11)
    if _is(u01, 0) and _is(u10, 0):
        if not _is(u00, 1):
            a.mul_(u00)
        if not _is(u11, 1):
            b.mul_(u11)
        return
    if g.name == "X":
        t = a.clone()
        a.copy_(b)
        b.copy_(t)
        return
    na = u00 * a
    na += u01 * b
    b.mul_(u11)
    b += u10 * a
    a.copy_(na)


def _pauli_string(psi, n, ops):
    out = psi.clone()
    for q, p in ops:
        a, b = _slice(out, n, {q: 0}), _slice(out, n, {q: 1})
        if p == "Z":
            b.neg_()
        else:
            t = a.clone()
            a.copy_(b if p == "X" else -1j * b)
            b.copy_(t if p == "X" else 1j * t)
    return out


def _observable(psi, n, terms):
    """O psi: the diagonal strings as one signed sum, the others one by one."""
    weight = torch.zeros(1, 1 << n, dtype=torch.float64, device="cuda")
    for c, ops in terms:
        if all(p == "Z" for _, p in ops):
            vals = {q: 0 for q, _ in ops}
            for bits in range(1 << len(ops)):
                v = {q: (bits >> k) & 1 for k, q in enumerate(vals)}
                _slice(weight, n, v).add_(c * (-1) ** bin(bits).count("1"))
    out = weight * psi
    for c, ops in terms:
        if not all(p == "Z" for _, p in ops):
            out += c * _pauli_string(psi, n, ops)
    return out


def _inner(a, b):
    """Re and Im of <a|b> for each register."""
    return torch.view_as_complex((torch.stack([(a.real * b.real + a.imag * b.imag).sum(-1),
                                               (a.real * b.imag - a.imag * b.real).sum(-1)], -1)))


def _zero(registers, n):
    psi = torch.zeros(registers, 1 << n, dtype=torch.complex128, device="cuda")
    psi[:, 0] = 1
    return psi


def _forward(psi, n, gates, params=None):
    for g in gates:
        _apply(psi, n, g, params[..., g.param] if g.param is not None else g.theta)
    return psi


def _gradient(psi, n, gates, params, terms):
    """Energies [R] and gradients [R, P] by walking the circuit backwards from its output; psi becomes its input."""
    lam = _observable(psi, n, terms)
    energy = _inner(psi, lam).real
    grad = torch.zeros(psi.shape[0], params.shape[-1], dtype=torch.float64, device="cuda")
    for g in reversed(gates):
        theta = params[..., g.param] if g.param is not None else g.theta
        if g.param is not None:  # U = exp(-i theta P / 2): the derivative is Im <lambda|P psi>
            x0, x1, l0, l1 = (_slice(v, n, {g.locs[0]: k}) for v in (psi, lam) for k in (0, 1))
            if g.name == "RZ":
                d = (l0.conj() * x0).imag - (l1.conj() * x1).imag
            else:
                d = (l0.conj() * x1).imag + (l1.conj() * x0).imag
            grad[:, g.param] += d.reshape(psi.shape[0], -1).sum(-1)
        _apply(psi, n, g, theta, dagger=True)
        _apply(lam, n, g, theta, dagger=True)
    return energy, grad


def _couplings(n, seed):
    """One coupling a bond (the XX, YY and ZZ of a bond share it), so that a matrix's values come from the seed."""
    j = W.rng(seed).uniform(0.5, 1.5, n)
    return np.repeat(j, 3)


def exact(case, seed):
    kind, n = case["kind"], case.get("n")
    if kind == "qft":
        psi = _random_amplitudes(n, case["dtype"], seed).to(torch.complex128).view(1, -1)
        return _forward(psi, n, W.qft(n, case["swaps"]))
    if kind == "vqe":
        gates, params = W.variational(n, case["depth"], _entangler(case), seed=seed)
        psi = _forward(_zero(1, n), n, gates, params)
        return psi, _inner(psi, _observable(psi, n, W.zz_chain(n))).real
    if kind == "gates":
        psi = _random_amplitudes(n, case["dtype"], seed).to(torch.complex128).view(1, -1)
        return _forward(psi, n, [g for _, g in W.single_gate_suite(n)])
    if kind == "batch":
        counts, gates, angles = _batch_inputs(case, seed)
        states, losses, grads = ([None] * len(counts) for _ in range(3))
        for k in gates:
            rows = [r for r, m in enumerate(counts) if m == k]
            params = torch.tensor(np.stack([angles[r] for r in rows]), device="cuda").double()
            psi = _forward(_zero(len(rows), k), k, gates[k], params)
            out = psi.clone()
            energy, grad = _gradient(psi, k, gates[k], params, W.zz_chain(k))
            for i, r in enumerate(rows):
                states[r], losses[r], grads[r] = out[i], energy[i], grad[i]
        return torch.cat(states), torch.stack(losses), torch.cat(grads)
    if kind == "train":
        gates, _ = W.variational(n, case["depth"], "ring", params=())
        params = torch.tensor(_angles(3 * n * case["depth"], seed, np.float32)).double()
        energy, grad = _gradient(_forward(_zero(1, n), n, gates, params), n, gates, params, W.tfim(n))
        return energy[0], grad[0]
    if kind == "brickwork":
        gates, params = W.brickwork(n, case["depth"], seed=seed)
        params = torch.tensor(params)
        psi = _forward(_zero(1, n), n, gates, params)
        energy, grad = _gradient(psi, n, gates, params, W.z_on(0))
        return energy[0], grad[0], psi
    if kind == "observe":
        psi = _random_amplitudes(n, case["dtype"], seed).to(torch.complex128).view(1, -1)
        return _inner(psi, _observable(psi, n, W.tfim(n))).real, None
    if kind == "matrix":
        x = torch.arange(1 << n, device="cuda")
        cols, vals = [x], [torch.zeros(1 << n, dtype=torch.complex128, device="cuda")]
        for (i, j), c in zip([(b, (b + 1) % n) for b in range(n)], _couplings(n, seed)[::3]):
            differ = ((x >> i) ^ (x >> j)) & 1
            vals[0] += c * (1 - 2 * differ).double()
            cols.append(x ^ ((1 << i) | (1 << j)))
            vals.append(2 * c * differ.to(torch.complex128))
        cols, vals = torch.stack(cols, 1), torch.stack(vals, 1)
        cols, order = cols.sort(1)
        vals = vals.gather(1, order)
        return None, None, vals[vals != 0]
    gates, params, uniforms = _shot_inputs(case, seed)
    shift = torch.eye(len(params), dtype=torch.float64, device="cuda") * (math.pi / 2)
    shifted = torch.tensor(params, device="cuda") + torch.stack([shift, -shift], 1).view(-1, len(params))
    psi = _forward(_zero(len(shifted), n), n, gates, shifted)
    energy = torch.zeros(len(shifted), dtype=torch.float64, device="cuda")
    for basis, u in zip("ZX", torch.tensor(uniforms, device="cuda")):  # the groups in the order of W.tfim's terms
        if basis == "X":
            for q in range(n):
                _apply(psi, n, W.Gate("H", (q,)))
        total = (psi.real ** 2 + psi.imag ** 2).cumsum(1)
        x = torch.searchsorted(total, u * total[:, -1:], right=True).clamp_(max=(1 << n) - 1)
        for c, ops in W.tfim(n):
            if ops[0][1] == basis:
                parity = sum((x >> q) & 1 for q, _ in ops) & 1
                energy += c * (1 - 2 * parity).double().mean(1)
    return 0.5 * (energy[0::2] - energy[1::2])
