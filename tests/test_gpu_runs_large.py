"""Runs of diagonal gates and of swaps on states of many tiles: every amplitude to a few roundings of its
own size, and bit for bit where amplitudes only move."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _state(n, dtype, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    v = torch.randn((1 << n, 2), generator=g, device="cuda", dtype=torch.float32 if dtype == 0 else torch.float64)
    return torch.view_as_complex(v * 2.0 ** (-n / 2))


def _apply(sv, n, dtype, gates, psi):
    import torch
    out = psi.clone()
    s = sv.sv_alloc(n, dtype, dev_buf=out, stream=torch.cuda.current_stream())
    sv.sv_set_state(s, psi)
    rep = sv.sv_apply_circuit(s, sv.sv_fuse(gates, n, 0))
    sv.sv_sync(s)
    s.free()
    return out, rep


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,top", [(22, 22), (25, 25), (25, 11)])      # top 11: inside the low bits
def test_diagonal_runs(gpu, dtype, n, top):
    import torch
    sv = gpu
    rng = np.random.default_rng(n + top)
    psi = _state(n, dtype, n)
    gates = []
    for i in range(30):
        k = int(rng.integers(1, 6))
        tg = tuple(int(t) for t in rng.choice(top, size=k, replace=False))
        d = np.exp(1j * rng.uniform(0, 6, 1 << k))
        if i % 2:
            d[: 1 << (k - 1)] = 1.0
        gates.append((tg, np.diag(d)))
    got, rep = _apply(sv, n, dtype, gates, psi)
    assert rep["bytes"] < 20 * 2 * psi.numel() * psi.element_size()     # gate by gate: about 22 states
    want = psi.to(torch.complex128)
    size = want.abs()
    k = torch.arange(1 << n, device="cuda", dtype=torch.int64)
    for tg, u in gates:
        l = sum(((k >> t) & 1) << j for j, t in enumerate(tg))
        want *= torch.from_numpy(np.ascontiguousarray(np.diag(u))).cuda()[l]
    # a rounded factor and a rounded product per gate, each at most 2 eps of the modulus
    eps = float(np.finfo(np.float32 if dtype == 0 else np.float64).eps)
    assert bool(torch.all((got - want).abs() <= 4 * len(gates) * eps * size))


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n", [23, 26])
def test_swap_runs(gpu, dtype, n):
    import torch
    sv = gpu
    rng = np.random.default_rng(n)
    swap = np.eye(4, dtype=np.complex128)[[0, 2, 1, 3]]
    psi = _state(n, dtype, n)
    p = [int(q) for q in rng.permutation(n)]
    for pairs in ([(i, n - 1 - i) for i in range(n // 2)], [(p[2 * i], p[2 * i + 1]) for i in range(n // 2)],
                  [(n - 1, n - 2), (n - 3, n - 4), (n - 5, n - 6)], [(0, 1), (2, 3), (4, n - 7)]):
        got, rep = _apply(sv, n, dtype, [(q, swap) for q in pairs], psi)
        assert rep["bytes"] == 2 * psi.numel() * psi.element_size()
        order = list(range(n))
        for a, b in pairs:
            order[a], order[b] = order[b], order[a]
        k = torch.arange(1 << n, device="cuda", dtype=torch.int64)
        src = torch.zeros_like(k)
        for a, b in enumerate(order):
            src |= ((k >> a) & 1) << b
        assert torch.equal(torch.view_as_real(got), torch.view_as_real(psi[src]))
