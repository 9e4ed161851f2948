"""Pauli sums through the many-terms-per-read kernels: Z strings inside, above and across the
tile, X and Y on every position, odd and even Y counts, more terms than one pass takes, states
smaller than a tile; against the oracle, and term by term against the general kernels
(sv_expect_noalloc)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _state(n, dtype, rng):
    v = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)) * np.exp2(rng.integers(-6, 1, 1 << n))
    v /= np.linalg.norm(v)
    return v.astype(np.complex64 if dtype == 0 else np.complex128)


def _mask(n, k, rng):
    return sum(1 << int(q) for q in rng.choice(n, size=min(k, n), replace=False))


def _terms(n, rng):
    z = [0] + [3 << i for i in range(n - 1)] + [(1 << i) | (1 << (n - 1)) for i in range(0, n - 1, 2)]
    z += [_mask(n, int(rng.integers(1, n + 1)), rng) for _ in range(12)]
    x = [0] * len(z)
    for i in range(n):                                           # X, Y and X with a Z string
        x += [1 << i] * 3
        z += [0, 1 << i, _mask(n, 3, rng) & ~(1 << i)]
    for i in range(n - 1):                                       # XX + YY
        x += [3 << i] * 2
        z += [0, 3 << i]
    for k in (3, 4, 5, n):                                       # wider flips; five and more: general kernel
        if k <= n:
            m = _mask(n, k, rng)
            x += [m] * 2
            z += [_mask(n, 4, rng), m]
    x += [1 << (n - 1)] * 6                                      # more than four terms of one X-part
    z += [_mask(n, 2, rng) for _ in range(6)]
    return x, z, [float(v) for v in rng.normal(size=len(x))]


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 11, 12, 13, 14, 17])
def test_pauli_sums_against_the_oracle(gpu, dtype, n):
    sv = gpu
    import torch
    rng = np.random.default_rng(60 + n)
    psi = _state(n, dtype, rng)
    s = sv.sv_alloc(n, dtype, stream=torch.cuda.current_stream())
    sv.sv_set_state(s, psi)
    x, z, c = _terms(n, rng)
    ref = psi.astype(np.complex128)
    each = [oracle.expect_pauli(ref, a, b).real for a, b in zip(x, z)]
    want = float(np.dot(c, each))
    # complex64: the products are FP32 (2^-24 of |psi_k||psi_l|, whose sum is at most 1) in
    # runs of eight: 2^-21 per term; complex128: 2^-45 per term
    tol = 2.0 ** (-21 if dtype == 0 else -45)
    assert abs(sv.sv_expect(s, x, z, c) - want) < tol * sum(abs(v) for v in c)
    for i in range(0, len(x), 7):                                # single terms
        assert abs(sv.sv_expect(s, [x[i]], [z[i]], [1.0]) - each[i]) < tol, (hex(x[i]), hex(z[i]))
    s.free()


def test_many_strings_take_several_passes(gpu):
    """700 Z strings with more mixed classes than a pass takes, and 60 single flips."""
    sv = gpu
    n, rng = 16, np.random.default_rng(8)
    psi = _state(n, 0, rng)
    s = sv.sv_alloc(n, 0)
    sv.sv_set_state(s, psi)
    z = [int(v) for v in rng.integers(0, 1 << n, 700)] + [int(v) for v in rng.integers(0, 1 << n, 60)]
    x = [0] * 700 + [1 << int(rng.integers(0, n)) for _ in range(60)]
    c = [float(v) for v in rng.normal(size=len(x))]
    got, want = sv.sv_expect(s, x, z, c), oracle.expect(psi.astype(np.complex128), x, z, c)
    assert abs(got - want) < 2.0 ** -21 * sum(abs(v) for v in c)
    s.free()


@pytest.mark.parametrize("dtype", [0, 1])
def test_special_amplitudes(gpu, dtype):
    """A basis state, the zero state, and an infinite amplitude (an infinite <Z0>, not NaN)."""
    sv = gpu
    n = 13
    s = sv.sv_alloc(n, dtype)
    sv.sv_set_basis(s, 5)
    assert sv.sv_expect(s, [0, 0], [1, 2], [1.0, 1.0]) == 0.0            # <Z0> = -1, <Z1> = 1
    assert sv.sv_expect(s, [1, 0], [0, 0], [3.0, 2.0]) == 2.0
    sv.sv_set_zero(s)
    assert sv.sv_expect(s, [0, 2], [1, 0], [1.0, 1.0]) == 0.0
    psi = np.zeros(1 << n, dtype=np.complex64 if dtype == 0 else np.complex128)
    psi[4] = np.inf
    sv.sv_set_state(s, psi)
    assert sv.sv_expect(s, [0], [1], [1.0]) == np.inf
    s.free()


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,count", [(3, 5), (11, 400), (13, 7), (15, 33)])
def test_batch_energies(gpu, dtype, n, count):
    """Z strings (inside, above and across a tile) and strings with X and Y, for every state."""
    sv = gpu
    import torch
    import workloads as W
    rng = np.random.default_rng(n)
    fam = [W.hea(n, 2, rng=rng) for _ in range(min(count, 9))]
    fused = [sv.sv_fuse(sv.gates_from_specs(f), n, 3) for f in fam]
    b = sv.sv_batch_alloc(n, dtype, count, stream=torch.cuda.current_stream())
    sv.sv_batch_apply(b, [fused[i % len(fused)] for i in range(count)])
    z = [0] + [3 << i for i in range(n - 1)] + [int(v) for v in rng.integers(0, 1 << n, 40)] + [1, 0, 5]
    x = [0] * (len(z) - 3) + [1, 1 << (n - 1), 3]
    c = [float(v) for v in rng.normal(size=len(z))]
    got = sv.sv_batch_expect(b, x, z, c)
    tol = (2.0 ** -21 if dtype == 0 else 2.0 ** -45) * sum(abs(v) for v in c)
    for i in list(range(min(count, 9))) + [count - 1]:
        psi = sv.sv_batch_get_state(b, i).astype(np.complex128)
        assert abs(got[i] - oracle.expect(psi, x, z, c)) < tol, i
    b.free()
