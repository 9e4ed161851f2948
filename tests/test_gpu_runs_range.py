"""Diagonal gates whose product leaves the state's range, one after the other in a circuit: the same
amplitudes as gate by gate, where zeros stay zero and every step is in range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("qubits", [(0, 1, 2, 3), (0, 5, 13, 9), (13, 12, 11, 4)])     # low bits, mixed, high
@pytest.mark.parametrize("sign", [1, -1])
def test_products_out_of_range(gpu, dtype, qubits, sign):
    sv = gpu
    import torch
    n, rng = 14, np.random.default_rng(2)
    e = sign * (20 if dtype == 0 else 160)
    v = (rng.uniform(1, 2, 1 << n) + 1j * rng.uniform(1, 2, 1 << n)) * 10.0 ** (-1.5 * e)
    v[::3] = 0.0
    psi = v.astype(np.complex64 if dtype == 0 else np.complex128)
    assert np.all(np.isfinite(psi)) and np.all(psi[1::3] != 0)
    # 10^e twice with phases around them: each step in range, their product not
    f = [10.0 ** e, np.exp(0.4j), 10.0 ** e, np.exp(-0.7j)]
    gates = [((q,), np.diag([f[i], f[i]])) for i, q in enumerate(qubits)]
    out = []
    for whole in (False, True):
        s = sv.sv_alloc(n, dtype, stream=torch.cuda.current_stream())
        sv.sv_set_state(s, psi)
        if whole:
            sv.sv_apply_circuit(s, sv.sv_fuse(gates, n, 0))
        else:
            for g in gates:
                sv.sv_apply_gate(s, *g)
        out.append(sv.sv_get_state(s))
        s.free()
    assert np.all(np.isfinite(out[0])) and np.all(out[0][::3] == 0)
    # four products, each correctly rounded up to two ulps of its modulus
    tol = 16 * np.finfo(np.float32 if dtype == 0 else np.float64).eps
    assert np.all(np.abs(out[1].astype(np.complex128) - out[0]) <= tol * np.abs(out[0].astype(np.complex128)))
