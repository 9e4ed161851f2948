"""Expectations of unnormalised complex64 states whose probabilities fit FP32 while their sums do
not: single states and batches, Z strings and strings with X."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [False, True])
def test_sums_beyond_single_precision(gpu, batch):
    sv = gpu
    import torch
    n, rng = 13, np.random.default_rng(3)
    # |psi_k|^2 up to 1.8e37 (eight of them below 3.4e38), 8192 of them about 1e41
    psi = (rng.uniform(-3e18, 3e18, 1 << n) + 1j * rng.uniform(-3e18, 3e18, 1 << n)).astype(np.complex64)
    z = [0, 1, 1 << (n - 1), 3 << 11, 5, 0]
    x = [0, 0, 0, 0, 0, 1 << 4]
    c = [1.0, 0.5, -0.25, 0.125, 2.0, 0.5]
    want = oracle.expect(psi.astype(np.complex128), x, z, c)
    if batch:
        buf = torch.zeros(2 << n, dtype=torch.complex64, device="cuda")
        b = sv.sv_batch_alloc(n, 0, 2, dev_buf=buf, stream=torch.cuda.current_stream())
        buf.copy_(torch.from_numpy(np.concatenate([psi, psi * np.float32(1e-18)])))
        got = sv.sv_batch_expect(b, x, z, c)
        small = oracle.expect((psi * np.float32(1e-18)).astype(np.complex128), x, z, c)
        b.free()
        assert abs(got[1] - small) < 2.0 ** -21 * sum(abs(v) for v in c) * np.sum(np.abs(psi * 1e-18) ** 2)
        got = got[0]
    else:
        s = sv.sv_alloc(n, 0, stream=torch.cuda.current_stream())
        sv.sv_set_state(s, psi)
        got = sv.sv_expect(s, x, z, c)
        s.free()
    # FP32 products in FP32 runs of eight: 2^-21 of the norm per term
    norm = np.sum(np.abs(psi.astype(np.complex128)) ** 2)
    assert abs(got - want) < 2.0 ** -21 * sum(abs(v) for v in c) * norm
