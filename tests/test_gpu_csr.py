"""The sparse matrix of a Pauli sum against its definition, entry by entry and bit by
bit: entry (i, i ^ x) is the sum, in the terms' order, of the terms of mask x; exact
zeros are not stored.  Registers below, at and above the sizes where a block of rows
and the segments of the rows begin; groups with and without a table of values, real
and complex; one mask and 64."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def parity(v):
    v = v.copy()
    for s in (32, 16, 8, 4, 2, 1):
        v ^= v >> s
    return v & 1


def reference(n, terms):
    i = np.arange(1 << n, dtype=np.int64)
    groups = {}
    for c, ops in terms:
        x = sum(1 << l for l, p in ops if p in "XY")
        z = sum(1 << l for l, p in ops if p in "ZY")
        k = bin(x & z).count("1") & 3
        groups.setdefault(x, []).append((c * (1, 0, -1, 0)[k], c * (0, 1, 0, -1)[k], z))
    cols, vals = [], []
    for x, members in groups.items():
        j = i ^ x
        re, im = np.zeros(1 << n), np.zeros(1 << n)
        for cr, ci, z in members:
            s = 1.0 - 2.0 * parity(j & z)
            re, im = re + s * cr, im + s * ci
        cols.append(j)
        vals.append(re + 1j * im)
    if not cols:
        return np.zeros(i.size + 1, np.int64), np.zeros(0, np.int64), np.zeros(0, complex)
    cols, vals = np.stack(cols, 1), np.stack(vals, 1)
    order = np.argsort(cols, axis=1)
    cols, vals = np.take_along_axis(cols, order, 1), np.take_along_axis(vals, order, 1)
    keep = vals != 0
    return np.concatenate([[0], keep.sum(1).cumsum()]), cols[keep], vals[keep]


def random_terms(n, count, seed, width):
    rs = W.rng(seed)
    return [(float(rs.integers(-2, 3)) / 2 + (0.1 if rs.random() < 0.3 else 0.0),
             tuple((int(l), "XYZ"[rs.integers(3)]) for l in rs.permutation(n)[: rs.integers(0, min(n, width) + 1)]))
            for _ in range(count)]


def observables(n):
    yield []
    yield [(2.0, ())]
    yield W.heisenberg(n) if n > 1 else W.tfim(n)
    yield [(c * (0.5 + 0.01 * k), ops) for k, (c, ops) in enumerate(W.tfim(n))][::-1]
    yield random_terms(n, 40, n, 3)
    # groups above the table's size with Y factors; cancelling copies
    yield [(0.3 * k, ((0, "Y"),) + tuple((l, "Z") for l in range(1, n) if (k >> (l % 5)) & 1)) for k in range(20)]
    yield [(s * 0.7, ((0, "X"), (n - 1, "Z")) if n > 1 else ((0, "X"),)) for s in (1, -1, 1, -1)]
    if n >= 6:  # 64 masks
        yield [(1.0 + k, tuple((l, "X") for l in range(6) if (k >> l) & 1)) for k in range(64)]


@pytest.mark.parametrize("n", [1, 2, 5, 6, 9, 10, 11, 13, 17, 18])
def test_csr_equals_its_definition(n):
    from paper_1912_10877_gb300 import qsim
    for k, terms in enumerate(observables(n)):
        rowptr, cols, vals = (v.cpu().numpy() for v in qsim.observable_csr(qsim.Observable(terms), n))
        rp, c, v = reference(n, terms)
        assert np.array_equal(rowptr, rp), k
        assert np.array_equal(cols, c), k
        assert np.array_equal(vals, v), k
