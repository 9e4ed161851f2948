"""Fields of single flips (X on every qubit, with and without Z elsewhere), whose passes keep their
sums in registers: one to many tiles, partly filled register sets, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n", [4, 7, 12, 13, 18, 20])
@pytest.mark.parametrize("zs", [0, 1])
def test_fields(gpu, dtype, n, zs):
    sv = gpu
    import torch
    rng = np.random.default_rng(n)
    v = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi = (v / np.linalg.norm(v)).astype(np.complex64 if dtype == 0 else np.complex128)
    s = sv.sv_alloc(n, dtype, stream=torch.cuda.current_stream())
    sv.sv_set_state(s, psi)
    x = [1 << i for i in range(n)]
    z = [zs << ((i + n // 2) % n) for i in range(n)]
    c = [float(u) for u in rng.normal(size=n)]
    want = oracle.expect(psi.astype(np.complex128), x, z, c)
    # FP32 products in runs of eight: 2^-21 of the norm (1) per term; complex128 2^-45
    assert abs(sv.sv_expect(s, x, z, c) - want) < 2.0 ** (-21 if dtype == 0 else -45) * sum(abs(u) for u in c)
    s.free()
