"""complex64 tensor-core passes whose targets include the lowest index bits (16-byte accesses when
bits 0-3 are targets), with one to many tiles per SM, as single states and as batches."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _groups(n, targets):
    """index[g, c]: the index of member c of group g."""
    free = [b for b in range(n) if b not in targets]
    g = np.arange(1 << len(free))
    base = sum((((g >> i) & 1) << b) for i, b in enumerate(free))
    c = np.arange(32)
    return base[:, None] + sum((((c >> i) & 1) << b) for i, b in enumerate(targets))[None, :]


def _inputs(n, rng):
    # rows of different scales
    v = (rng.uniform(-1, 1, 1 << n) + 1j * rng.uniform(-1, 1, 1 << n)) * np.exp2(rng.integers(-12, 1, 1 << n))
    return v.astype(np.complex64), (rng.uniform(-1, 1, (32, 32)) + 1j * rng.uniform(-1, 1, (32, 32))) / 8


def _check(got, psi, idx, u):
    al = psi[idx].astype(np.complex128)
    want = al @ u.T
    # a row of components up to M, entries up to R, 64 products per component: the operands' slices
    # 64 x 2 x 2^-26 M R, the dropped slice products 64 x 2 x 2^-27 x 4 M R, the truncation of D12
    # 16 x 2^-9 x 4 x 2^-16 M R, FP32 rounding of the output 2 x 2^-24 x 64 M R: below 2^-16 M R
    m = np.maximum(np.abs(al.real), np.abs(al.imag)).max(axis=1, keepdims=True)
    r = max(np.abs(u.real).max(), np.abs(u.imag).max())
    d = got[idx] - want
    assert np.all(np.abs(d.real) <= 2.0 ** -16 * m * r) and np.all(np.abs(d.imag) <= 2.0 ** -16 * m * r)


@pytest.mark.parametrize("n", [13, 15, 23])
@pytest.mark.parametrize("targets", [(0, 1, 2, 3, 4), (0, 1, 2, 3, -1), (0, 1, 2, 4, 5), (1, 2, 3, 4, 5), (0, -4, -3, -2, -1)])
def test_low_targets(gpu, n, targets):
    import torch
    sv = gpu
    targets = tuple(t % n for t in targets)
    psi, u = _inputs(n, np.random.default_rng(n))
    s = sv.sv_alloc(n, 0, stream=torch.cuda.current_stream())
    sv.sv_set_state(s, psi)
    sv.sv_apply_gate(s, targets, u)
    got = sv.sv_get_state(s)
    s.free()
    _check(got, psi, _groups(n, targets), u)


@pytest.mark.parametrize("targets", [(0, 1, 2, 3, 4), (0, 1, 2, 3, 12), (0, 1, 5, 6, 7)])
def test_low_targets_in_a_batch(gpu, targets):
    import torch
    sv = gpu
    n, count, rng = 13, 170, np.random.default_rng(4)
    pairs = [_inputs(n, rng) for _ in range(3)]
    buf = torch.zeros(count << n, dtype=torch.complex64, device="cuda")
    b = sv.sv_batch_alloc(n, 0, count, dev_buf=buf, stream=torch.cuda.current_stream())
    buf.copy_(torch.from_numpy(np.concatenate([pairs[i % 3][0] for i in range(count)])))
    sv.sv_batch_apply(b, [sv.sv_fuse([(targets, pairs[i % 3][1])], n, 5) for i in range(count)])
    idx = _groups(n, targets)
    for i in (0, 1, 2, 77, count - 1):
        _check(sv.sv_batch_get_state(b, i), pairs[i % 3][0], idx, pairs[i % 3][1])
    b.free()
