"""Expectation sums against the oracle at the edges of their kernels: registers
below, at and above a step, a chunk and a block; more Z strings and more x masks than
one launch takes; several terms of one mask; a register on an 8-byte boundary.  Both
sides read the same stored amplitudes; the sums' rounding is below (64 + log2 of the
pair count) 2^-53 of sum |c|, held here to 1e-13 of it."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

TDT = {"c64": torch.complex64, "c128": torch.complex128}


def random_terms(n, count, seed, letters="XYZ"):
    rs = W.rng(seed)
    out = []
    for _ in range(count):
        q = rs.permutation(n)[: rs.integers(0, min(n, 4) + 1)]
        out.append((float(rs.standard_normal()), tuple((int(l), letters[rs.integers(len(letters))]) for l in q)))
    return out


def observables(n):
    yield random_terms(n, 30, 3 * n)
    yield W.tfim(n)
    yield W.heisenberg(n)
    yield random_terms(n, 150, n, "Z")                                   # several launches of Z strings
    yield [(0.5 + l, ((l, p),)) for l in range(n) for p in "XY"] * 3      # six terms of each mask
    yield [(1.0, ((a, "X"), (b, "Y"))) for a in range(n) for b in range(n) if a != b]


@pytest.mark.parametrize("dt", ["c64", "c128"])
@pytest.mark.parametrize("n,nreg", [(1, 3), (2, 2), (5, 70), (9, 2), (10, 1), (11, 2), (13, 1), (14, 2), (15, 1), (17, 1)])
def test_expectations_equal_the_oracles(dt, n, nreg):
    from paper_1912_10877_gb300 import qsim
    st = qsim.State(n, dtype=TDT[dt], nbatch=nreg)
    st.upload(np.concatenate([W.haar_state(n, seed=r + 5 * n) for r in range(nreg)]))
    amps = st.numpy().astype(np.complex128).reshape(nreg, -1)
    for k, terms in enumerate(observables(n)):
        if n == 1 and k in (2, 5):
            continue
        got = st.expect(qsim.Observable(terms))
        for r in {0, nreg - 1}:
            want = oracle.expect(amps[r], n, terms)
            assert abs(got[r] - want) < 1e-13 * sum(abs(c) for c, _ in terms), (k, r, got[r], want)


def test_static_expectation_of_a_register_on_an_8_byte_boundary():
    from paper_1912_10877_gb300 import _native as N
    n = 12
    psi = W.haar_state(n, seed=2).astype(np.complex64)
    buf = torch.zeros((1 << n) + 1, dtype=torch.complex64, device="cuda")
    buf[1:] = torch.from_numpy(psi)
    assert buf[1:].data_ptr() % 16 == 8
    terms = random_terms(n, 40, 11)
    arr = (N.PauliTerm * len(terms))()
    for i, (c, ops) in enumerate(terms):
        arr[i].coeff = c
        arr[i].x_mask = sum(1 << l for l, p in ops if p in "XY")
        arr[i].z_mask = sum(1 << l for l, p in ops if p in "ZY")
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    N.check(N.lib().qs_expect_static(ctypes.c_void_p(buf.data_ptr() + 8), N.QS_C64, n, 1, arr, len(terms),
                                     ctypes.c_void_p(out.data_ptr()),
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    want = oracle.expect(psi.astype(np.complex128), n, terms)
    assert abs(float(out.item()) - want) < 1e-13 * sum(abs(c) for c, _ in terms)
