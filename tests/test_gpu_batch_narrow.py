"""Batched complex64 gates of one to three qubits: every group of 2^k amplitudes keeps FP32 accuracy
relative to its own size whatever its neighbours hold, and an infinity stays in its group."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9, 13, 15])
@pytest.mark.parametrize("targets", [(3,), (8,), (0, 6), (2, 5, 7)])
def test_groups_keep_their_own_accuracy(gpu, n, targets):
    import torch
    sv = gpu
    k, count = len(targets), 3
    d = 1 << k
    rng = np.random.default_rng(10 * n + k)
    free = [b for b in range(n) if b not in targets]
    g = np.arange(1 << len(free))
    base = sum((((g >> i) & 1) << b) for i, b in enumerate(free))
    idx = base[:, None] + sum((((np.arange(d) >> i) & 1) << b) for i, b in enumerate(targets))[None, :]
    psi = (rng.uniform(-1, 1, (count, 1 << n)) + 1j * rng.uniform(-1, 1, (count, 1 << n))).astype(np.complex64)
    for s in range(count):                               # groups from 1 down to 2^-80
        psi[s][idx] *= np.exp2(-rng.integers(0, 81, idx.shape[0]))[:, None].astype(np.float32)
    psi[1][idx[5, 0]] = np.inf
    u = [np.linalg.qr(rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d)))[0] for _ in range(count)]
    buf = torch.zeros(count << n, dtype=torch.complex64, device="cuda")
    b = sv.sv_batch_alloc(n, 0, count, dev_buf=buf, stream=torch.cuda.current_stream())
    buf.copy_(torch.from_numpy(psi.reshape(-1)))
    sv.sv_batch_apply(b, [sv.sv_fuse([(targets, m)], n, 0) for m in u])
    # 2^(k+1) products per component: rounded entries and a chain of fused multiply-adds
    tol = (2 * d + 2) * 2.0 ** -24
    for s in range(count):
        got = sv.sv_batch_get_state(b, s).astype(np.complex128)[idx]
        a = psi[s].astype(np.complex128)[idx]
        ok = np.all(np.isfinite(a), axis=1)
        assert np.sum(~ok) == (1 if s == 1 else 0)
        want, size = a[ok] @ u[s].T, np.abs(a[ok]) @ np.abs(u[s]).T * np.sqrt(2)
        diff = got[ok] - want
        assert np.all(np.isfinite(got[ok]))
        assert np.all(np.abs(diff.real) <= tol * size) and np.all(np.abs(diff.imag) <= tol * size)
    b.free()
