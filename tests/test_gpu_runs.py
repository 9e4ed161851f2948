"""Runs of diagonal gates and of swaps that share one pass: against the oracle, against the same
schedule with every gate dense, and bit for bit where nothing changes."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
TOL = {0: 1e-5, 1: 1e-12}     # the library's stated max-abs amplitude errors


def _torch():
    import torch
    return torch


def _state(n, dtype, rng):
    v = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    return (v / np.linalg.norm(v)).astype(np.complex64 if dtype == 0 else np.complex128)


def _apply(sv, n, dtype, gates, psi, policy=0):
    s = sv.sv_alloc(n, dtype, stream=_torch().cuda.current_stream())
    sv.sv_set_policy(s, policy)
    sv.sv_set_state(s, psi)
    rep = sv.sv_apply_circuit(s, sv.sv_fuse(gates, n, 0))
    out = sv.sv_get_state(s)
    s.free()
    return out, rep


def _diagonals(n, count, rng, low):
    """Phases on random qubits (`low`: most of them below bit 13, so that the run's low qubits
    connect and it has to end), some with entries exactly 1."""
    gates = []
    for i in range(count):
        k = int(rng.integers(1, 6))
        pool = np.arange(min(n, 13)) if low and i % 3 else np.arange(n)
        tg = tuple(int(t) for t in rng.choice(pool, size=k, replace=False))
        d = np.exp(1j * rng.uniform(0, 6, 1 << k))
        if i % 2:
            d[: 1 << (k - 1)] = 1.0                      # controlled on the highest local bit
        gates.append((tg, np.diag(d)))
    return gates


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,low", [(13, True), (14, False), (16, True), (19, False)])
def test_diagonal_runs(gpu, dtype, n, low):
    rng = np.random.default_rng(100 + n)
    psi = _state(n, dtype, rng)
    gates = _diagonals(n, 60, rng, low)
    got, rep = _apply(gpu, n, dtype, gates, psi)
    ref = oracle.run(psi.astype(np.complex128), gates)
    assert np.max(np.abs(got - ref)) < TOL[dtype]
    assert rep["passes"] == len(gates)
    assert rep["bytes"] < 30 * 2 * psi.nbytes           # the gates one by one: about 45 states


@pytest.mark.parametrize("dtype", [0, 1])
def test_amplitudes_with_factor_one_keep_their_bits(gpu, dtype):
    """Controls on every tile region: low bits, high bits and both; signed zeros and infinities
    outside the controlled part come back as they were."""
    rng = np.random.default_rng(3)
    n = 15
    psi = _state(n, dtype, rng)
    psi[::7] = -0.0
    psi[3] = np.inf                                     # bit 14 clear
    gates = [((c, 14), np.diag([1.0, 1.0, 1.0, np.exp(0.3j * (c + 1))])) for c in (0, 3, 7, 12, 13, 1, 5, 11)] * 2
    got, _ = _apply(gpu, n, dtype, gates, psi)
    half = 1 << 14
    u = np.uint32 if dtype == 0 else np.uint64
    assert np.array_equal(got[:half].view(u), psi[:half].view(u))
    ref = oracle.run(np.where(np.isfinite(psi), psi, 0).astype(np.complex128), gates)
    assert np.max(np.abs(got[half:] - ref[half:])) < TOL[dtype]


def _swap(a, b):
    return ((a, b), np.eye(4, dtype=np.complex128)[[0, 2, 1, 3]])


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n", [13, 14, 17, 20])
def test_swap_runs(gpu, dtype, n):
    rng = np.random.default_rng(200 + n)
    psi = _state(n, dtype, rng)
    p = [int(q) for q in rng.permutation(n)]
    cycle = np.zeros((8, 8), dtype=np.complex128)       # bits (0, 1, 2) -> (1, 2, 0)
    for c in range(8):
        cycle[((c << 1) | (c >> 2)) & 7, c] = 1.0
    runs = {
        "reversal": [_swap(i, n - 1 - i) for i in range(n // 2)],
        "random pairs": [_swap(p[2 * i], p[2 * i + 1]) for i in range(n // 2)],
        "high only": [_swap(n - 1, n - 2), _swap(n - 3, n - 4), _swap(n - 5, n - 6), _swap(n - 1, n - 2)],
        "low only": [_swap(0, 1), _swap(2, 3), _swap(4, 5)],
        "cycles": [_swap(0, 1), _swap(1, 2), _swap(2, n - 1), _swap(0, 1), _swap(1, 2), _swap(n - 1, 0)],
        "three-bit cycle": [((1, n - 1, 4), cycle)] * 3 + [((p[0], p[1], p[2]), cycle)] * 2,
    }
    for name, gates in runs.items():
        got, _ = _apply(gpu, n, dtype, gates, psi)
        want, _ = _apply(gpu, n, dtype, [], psi)
        ref = oracle.run(psi.astype(np.complex128), gates)
        assert np.array_equal(got, ref.astype(psi.dtype)), name    # moves only
        assert np.array_equal(want, psi)


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,k", [(13, 5), (14, 3), (17, 4), (20, 5)])
def test_qft(gpu, dtype, n, k):
    sv = gpu
    specs = W.qft(n)
    ref = oracle.simulate(n, specs, x=12345 % (1 << n))
    for policy in (0, sv.SV_POLICY_DENSE_ONLY):
        s = sv.sv_alloc(n, dtype, stream=_torch().cuda.current_stream())
        sv.sv_set_policy(s, policy)
        sv.sv_set_basis(s, 12345 % (1 << n))
        c = sv.sv_fuse(sv.gates_from_specs(specs), n, k)
        rep = sv.sv_apply_circuit(s, c)
        assert np.max(np.abs(sv.sv_get_state(s) - ref)) < TOL[dtype]
        s.free()
