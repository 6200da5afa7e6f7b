"""Several host threads, a handle each (include/qsim.h), on calls whose kernels take shared memory
by the call's size: no thread's launch depends on what another asked for."""
import ctypes
import threading

import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def together(jobs, repeats):
    """Runs every job `repeats` times in a thread of its own; the last results in order."""
    out, errors, start = [None] * len(jobs), [], threading.Barrier(len(jobs))

    def work(k):
        try:
            start.wait()
            for _ in range(repeats):
                out[k] = jobs[k]()
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    return out


def test_sparse_matrices_of_few_and_many_groups():
    from paper_1912_10877_gb300 import _native as N
    from paper_1912_10877_gb300 import qsim
    n = 8
    few = W.tfim(n)[:1]
    many = [(1.0 + k + 0.1 * j, tuple((l, "X") for l in range(6) if (k >> l) & 1) + ((6 + j % 2, "Z"),))
            for k in range(64) for j in range(4)]  # 64 groups without a table of values
    want, got, jobs = [], [], []
    for terms in (few, many):
        obs = qsim.Observable(terms)
        rowptr, cols, vals = qsim.observable_csr(obs, n)
        want.append((cols, vals))
        got.append((torch.zeros_like(cols), torch.zeros_like(vals)))
        args = [ctypes.c_void_p(t.data_ptr()) for t in (rowptr, *got[-1])]
        jobs.append(lambda o=obs, a=args, keep=rowptr: N.check(N.lib().qs_observable_csr_fill(o.handle, n, *a, None)))
    torch.cuda.synchronize()
    together(jobs, 5000)
    torch.cuda.synchronize()
    for g, w in zip(got, want):
        assert all(torch.equal(a, b) for a, b in zip(g, w))


def test_swap_passes_of_two_tile_sizes():
    from paper_1912_10877_gb300 import qsim
    n = 16
    psi = W.haar_state(n, seed=3).astype(np.complex64)
    networks = [[W.Gate("SWAP", (0, 1))], [W.Gate("SWAP", (10, 15))]]
    states = [qsim.State(n, dtype=torch.complex64).upload(psi) for _ in networks]
    circuits = [qsim.Circuit(g, n) for g in networks]
    jobs = [lambda s=s, c=c: s.apply_circuit(c, tiles=True) for s, c in zip(states, circuits)]
    together(jobs, 3001)
    for s, g in zip(states, networks):
        s.sync()
        assert np.array_equal(s.numpy().astype(np.complex128), oracle.apply_circuit(psi.astype(np.complex128), n, g))
