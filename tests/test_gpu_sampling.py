"""The sampler's routes against the oracle, index for index: registers below, at and
above a level-0 block (1024 amplitudes) and a level-1 block (2^20), with fewer and
more shots than level-0 blocks, one register and a batch."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def sparse_state(n, seed):
    """A state with long runs of zeros (blocks without weight, at both ends too)."""
    psi = W.haar_state(n, seed=seed)
    keep = W.rng(seed + 1).random(1 << n) < 0.01
    keep[: 1 << max(0, n - 2)] = False
    keep[-(1 << max(0, n - 3)):] = False
    keep[(1 << n) // 2] = True
    psi[~keep] = 0
    return psi


@pytest.mark.parametrize("dt", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("n,nreg,nshots", [(1, 3, 5), (4, 1, 1), (9, 40, 33), (10, 5, 300), (11, 3, 1), (11, 3, 2),
                                           (13, 7, 64), (14, 2, 15), (20, 1, 100), (20, 1, 2000), (21, 2, 50),
                                           (21, 1, 5000)])
def test_samples_equal_the_oracles(dt, n, nreg, nshots):
    from paper_1912_10877_gb300 import qsim
    u = W.shot_uniforms(nshots, seed=n, nreg=nreg)
    u[:, 0] = 0.0
    u[:, -1] = np.nextafter(1.0, 0.0)
    for make in (W.haar_state, sparse_state):
        psi = np.concatenate([make(n, seed=7 * n + r) for r in range(nreg)])
        st = qsim.State([n] * nreg, dtype=dt).upload(psi)
        amps = st.numpy().astype(np.complex128).reshape(nreg, -1)
        got = st.measure(u)
        for r in range(nreg):
            assert np.array_equal(got[r], oracle.sample(amps[r], n, u[r])), (make.__name__, r)


def test_register_without_weight():
    from paper_1912_10877_gb300 import qsim
    for n in (3, 12):
        st = qsim.State(n, dtype=torch.complex64).upload(np.zeros(1 << n))
        u = W.shot_uniforms(8, seed=1)
        assert np.array_equal(st.measure(u)[0], oracle.sample(np.zeros(1 << n, np.complex128), n, u[0]))


@pytest.mark.parametrize("dt", [torch.complex64, torch.complex128])
@pytest.mark.parametrize("n,nshots", [(9, 3), (12, 2), (12, 9), (21, 3)])
def test_targets_that_no_sum_may_exceed(dt, n, nshots):
    """A target of -0 (amplitudes without weight come first) and a NaN total of either sign: the
    contract's comparisons are those of floating-point numbers, on every route."""
    from paper_1912_10877_gb300 import qsim
    dim = 1 << n
    u = np.full(nshots, 0.5)
    u[0] = -0.0
    first = np.zeros(dim, np.complex128)
    first[5], first[dim - 3] = 0.6, 0.8
    states = [first]
    for nan in (np.nan, np.copysign(np.nan, -1.0)):
        for at in (2, dim // 2 + 1):
            psi = first.copy()
            psi[at] = complex(nan, 0.0)
            states.append(psi)
    for k, psi in enumerate(states):
        st = qsim.State(n, dtype=dt).upload(psi)
        got = st.measure(u[None])
        assert np.array_equal(got[0], oracle.sample(st.numpy().astype(np.complex128), n, u)), k


def test_device_without_room_for_the_running_sums():
    """128 MiB left on the device: the running sums of 2^25 probabilities do not fit (256 MiB),
    nor do 2^24 uniforms with their samples; the same samples as with room."""
    from paper_1912_10877_gb300 import qsim

    def amplitudes(st, seed):
        g = torch.Generator(device="cuda").manual_seed(seed)
        st.buffer.copy_(torch.randn(st.buffer.shape, dtype=st.buffer.dtype, device="cuda", generator=g))
        return st

    cases = [([25], 1 << 15), ([4] * 4096, 4096)]  # as many shots as level-0 blocks; many shots on many registers
    states = [amplitudes(qsim.State(sizes, dtype=torch.complex64), k) for k, (sizes, _) in enumerate(cases)]
    uniforms = [W.shot_uniforms(nshots, seed=k, nreg=len(sizes)) for k, (sizes, nshots) in enumerate(cases)]
    want = []
    for (sizes, _), st, u in zip(cases, states, uniforms):
        other = qsim.State(sizes, dtype=torch.complex64)
        other.buffer.copy_(st.buffer)
        other.measure(u[:, :2])  # the kernels of either route are loaded
        want.append(other.measure(u))
        del other
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - (128 << 20), dtype=torch.uint8, device="cuda")
    try:
        got = [st.measure(u) for st, u in zip(states, uniforms)]
    finally:
        del filler
        torch.cuda.empty_cache()
    for g, w in zip(got, want):
        assert np.array_equal(g, w)
