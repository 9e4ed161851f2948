"""Batched sums of Z strings that do not share tiled reads: coefficients keep more than FP32's digits in
complex64, and every pattern on the lowest index bits is taken, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def test_coefficients_are_not_rounded_to_single_precision(gpu):
    import torch
    sv = gpu
    n, count = 14, 40
    buf = torch.zeros((count, 1 << n), dtype=torch.complex64, device="cuda")
    b = sv.sv_batch_alloc(n, 0, count, dev_buf=buf, stream=torch.cuda.current_stream())
    buf.fill_(2.0 ** -7)                                  # every p = 2^-14
    # <1> = 1 and the others 0: their signed sums over eight amplitudes are exactly 0
    z = [0] + [1 + (i % 7) | (i + 1) << 12 for i in range(3)] + [5 | 64 * i for i in range(1, 9)]
    c = [0.1 + 1.0 / 3.0] + [1.0 / 7.0] * (len(z) - 1)
    got = sv.sv_batch_expect(b, [0] * len(z), z, c)
    # two floats keep 2^-48 of a coefficient; FP64 sums of equal terms
    assert np.max(np.abs(got - c[0])) < 2.0 ** -45
    b.free()


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n,count", [(1, 5), (2, 7), (3, 40), (9, 33), (15, 21)])
def test_unlike_strings(gpu, dtype, n, count):
    import torch
    sv = gpu
    rng = np.random.default_rng(n)
    psi = rng.normal(size=(count, 1 << n)) + 1j * rng.normal(size=(count, 1 << n))
    psi = (psi / np.linalg.norm(psi, axis=1)[:, None]).astype(np.complex64 if dtype == 0 else np.complex128)
    buf = torch.zeros((count, 1 << n), dtype=torch.complex64 if dtype == 0 else torch.complex128, device="cuda")
    b = sv.sv_batch_alloc(n, dtype, count, dev_buf=buf, stream=torch.cuda.current_stream())
    buf.copy_(torch.from_numpy(psi))
    z = [int(v) for v in rng.integers(0, 1 << n, 70)]
    c = [float(v) for v in rng.normal(size=len(z))]
    got = sv.sv_batch_expect(b, [0] * len(z), z, c)
    # per string: products and sums of eight in FP32, 32 strings added to a run: 2^-18 of the norm
    tol = (2.0 ** -18 if dtype == 0 else 2.0 ** -45) * sum(abs(v) for v in c)
    for i in (0, count // 2, count - 1):
        assert abs(got[i] - oracle.expect(psi[i].astype(np.complex128), [0] * len(z), z, c)) < tol
    b.free()
