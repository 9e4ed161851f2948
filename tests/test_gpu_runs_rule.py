"""Which diagonal gates share a pass on states where launches count: a few go one by one, many together
(the report's bytes tell), with the oracle's amplitudes either way."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["spread", "low"])
@pytest.mark.parametrize("dtype,n,m,run", [(0, 13, 2, False), (0, 19, 2, False), (0, 13, 3, True), (0, 20, 2, True),
                                           (0, 23, 2, True), (1, 13, 2, False), (1, 19, 2, False), (1, 14, 3, "low"),
                                           (1, 14, 4, True), (1, 20, 2, "low"), (1, 23, 3, True), (0, 15, 9, True),
                                           (1, 15, 9, True)])
def test_few_gates_on_small_states_go_one_by_one(gpu, dtype, n, m, run, where):
    import torch
    sv = gpu
    rng = np.random.default_rng(n + m)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dtype == 0 else np.complex128)
    gates = [((int(q),), np.diag(np.exp(1j * rng.uniform(0, 6, 2)))) for q in np.linspace(0, n - 1 if where == "spread" else 11, m)]
    s = sv.sv_alloc(n, dtype, stream=torch.cuda.current_stream())
    sv.sv_set_state(s, psi)
    rep = sv.sv_apply_circuit(s, sv.sv_fuse(gates, n, 0))
    got = sv.sv_get_state(s)
    s.free()
    assert rep["bytes"] == 2 * psi.nbytes * (1 if run in (True, where) else m)
    want = oracle.run(psi.astype(np.complex128), gates)
    # one rounded factor per gate and one rounded product each, of |z| relative to the amplitude
    eps = float(np.finfo(np.float32 if dtype == 0 else np.float64).eps)
    assert np.all(np.abs(got - want) <= 4 * (m + 1) * eps * np.abs(want))
