"""Pauli sums where every block walks over many tiles (its buffers refilled, its barriers' phases and
its tables of tile signs in turn, its sums moved on to FP64), on single states and on batches of more
states than the device holds blocks.  Amplitudes and coefficients are small integers, so every
product and partial sum is exact in both precisions and the results have to be equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _integers(shape, dtype, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    v = torch.randint(-7, 8, (*shape, 2), generator=g, device="cuda", dtype=torch.int8)
    return v, torch.view_as_complex(v.to(torch.float32 if dtype == 0 else torch.float64))


def _exact(v, n, x, z):
    """<psi| P |psi> of integer amplitudes v[..., 2^n, 2], in 64-bit integers."""
    import torch
    k = torch.arange(1 << n, device="cuda", dtype=torch.int32)

    def odd(m):
        w = k & m
        for s in (16, 8, 4, 2, 1):
            w = w ^ (w >> s)
        return w & 1
    p, q = v, v
    if x:
        q = v.index_select(v.dim() - 2, (k ^ x).to(torch.int64))
    a, b, c, d = (t.to(torch.int16) for t in (p[..., 0], p[..., 1], q[..., 0], q[..., 1]))
    y = bin(x & z).count("1") & 3                                # i^y times (re + i im): its real part
    part = (c * a + d * b) if y % 2 == 0 else (c * b - d * a)
    sign = (1 - 2 * odd(z).to(torch.int16)) * (1 if y in (0, 3) else -1)
    return (part * sign).sum(dim=-1, dtype=torch.int64)


def _terms(n, rng):
    low, top = 11, n - 1
    mixed = [(1 << top) | 5, (1 << top) | 9, (3 << (top - 1)) | 2]       # two signs on the high bits
    z = [0, 1, 3 << 4, 1 << low, 1 << top, 5 << (top - 2), 3 << (low - 1)] + [3 << i for i in range(n - 1)] + mixed
    x = [0] * len(z)
    for i in range(n):                                           # X, and Y or X with Z on some
        x.append(1 << i)
        z.append(0)
        if i % 3 == 0:
            x += [1 << i] * 2
            z += [1 << i, int(rng.integers(0, 1 << n)) & ~(1 << i)]
    for m in ((1 << top) | 1, (1 << top) | (1 << (top - 3)), 7, (1 << top) | (1 << low) | 6):
        x += [m, m]
        z += [m, int(rng.integers(0, 1 << n))]
    return x, z, [float(c) for c in rng.integers(-3, 4, len(x))]


@pytest.mark.parametrize("dtype,n", [(0, 22), (0, 29), (1, 21), (1, 24)])
def test_single_states(gpu, dtype, n):
    import torch
    sv = gpu
    rng = np.random.default_rng(n)
    v, psi = _integers((1 << n,), dtype, n)
    s = sv.sv_alloc(n, dtype, stream=torch.cuda.current_stream())
    sv.sv_set_state(s, psi)
    x, z, c = _terms(n, rng)
    each = [int(_exact(v, n, a, b)) for a, b in zip(x, z)]
    plain = [i for i in range(len(x)) if z[i] == 0]              # single flips (and 1) alone
    zs = [i for i in range(len(x)) if x[i] == 0]
    for pick in (range(len(x)), plain, zs, [4], [zs[-1]], [plain[1]]):
        got = sv.sv_expect(s, [x[i] for i in pick], [z[i] for i in pick], [c[i] for i in pick])
        assert got == sum(c[i] * each[i] for i in pick), (len(pick), got)
    if n <= 22:                                                  # the general kernels
        out = torch.zeros(1, dtype=torch.float64, device="cuda")
        sv.sv_expect_noalloc(psi, n, dtype, x, z, c, out, stream=torch.cuda.current_stream())
        assert float(out[0]) == sum(a * b for a, b in zip(c, each))
    s.free()


@pytest.mark.parametrize("dtype,n,count", [(0, 17, 320), (0, 21, 305), (1, 16, 310)])
def test_batches(gpu, dtype, n, count):
    import torch
    sv = gpu
    rng = np.random.default_rng(n)
    v, psi = _integers((count, 1 << n), dtype, n)
    b = sv.sv_batch_alloc(n, dtype, count, dev_buf=psi, stream=torch.cuda.current_stream())
    psi.copy_(torch.view_as_complex(v.to(torch.float32 if dtype == 0 else torch.float64)))   # it starts as |0>
    x, z, c = _terms(n, rng)
    pick = [i for i in range(len(x)) if x[i] == 0] + [len(x) - 1]
    x, z, c = ([t[i] for i in pick] for t in (x, z, c))
    want = np.zeros(count)
    for a, m, w in zip(x, z, c):
        want += w * np.concatenate([_exact(v[i:i + 32], n, a, m).cpu().numpy() for i in range(0, count, 32)])
    assert np.array_equal(sv.sv_batch_expect(b, x, z, c), want)
    b.free()
