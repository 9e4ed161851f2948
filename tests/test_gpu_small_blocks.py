"""Small circuits whose gates just fit, or just do not fit, the small and the large parameter block of the
many-gates launch, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


# 16 bytes per gate and 8 (complex64) or 16 per entry: 2 KiB hold 42 or 25 one-qubit gates, 28 KiB 597 or 358
@pytest.mark.parametrize("dtype,counts", [(0, (1, 42, 43, 597, 598)), (1, (1, 25, 26, 358, 359))])
@pytest.mark.parametrize("n", [3, 12])
def test_parameter_blocks(gpu, dtype, counts, n):
    import torch
    sv = gpu
    rng = np.random.default_rng(n)
    gates = [((int(rng.integers(0, n)),), np.array(W.haar_unitary(2, rng)).reshape(2, 2)) for _ in range(max(counts))]
    psi0 = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi0 = (psi0 / np.linalg.norm(psi0)).astype(np.complex64 if dtype == 0 else np.complex128)
    eps = float(np.finfo(np.float32 if dtype == 0 else np.float64).eps)
    for m in counts:
        s = sv.sv_alloc(n, dtype, stream=torch.cuda.current_stream())
        sv.sv_set_state(s, psi0)
        sv.sv_apply_circuit(s, sv.sv_fuse(gates[:m], n, 0))
        got = sv.sv_get_state(s)
        s.free()
        want = oracle.run(psi0.astype(np.complex128), gates[:m])
        # a gate adds at most 4 eps of the state's norm (1) to the error vector: two rounded entries and
        # a chain of four fused multiply-adds per row
        assert np.linalg.norm(got - want) <= 4 * (m + 1) * eps, m
