"""The search for runs costs host time in proportion to the gates: a long circuit of structured gates
that share nothing takes as long as its pieces one after the other."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["permutations", "phases"])
def test_long_circuits_cost_as_much_as_their_pieces(gpu, kind):
    import torch
    sv = gpu
    n, count, piece = 13, 40000, 400
    rng = np.random.default_rng(0)
    if kind == "permutations":
        u = np.eye(4, dtype=np.complex128)[[0, 3, 2, 1]]             # CNOT
        gates = [(tuple(int(q) for q in rng.choice(n, size=2, replace=False)), u) for _ in range(count)]
    else:                                                             # a 32nd of the state each
        u = np.diag([1.0] * 31 + [np.exp(0.1j)])
        gates = [(tuple(int(q) for q in rng.choice(n, size=5, replace=False)), u) for _ in range(count)]
    whole = [sv.sv_fuse(gates, n, 0)]
    pieces = [sv.sv_fuse(gates[i:i + piece], n, 0) for i in range(0, count, piece)]
    s = sv.sv_alloc(n, 1, stream=torch.cuda.current_stream())
    best = []
    for circuits in (whole, pieces):
        times = []
        for _ in range(3):
            sv.sv_sync(s)
            t = time.perf_counter()
            for c in circuits:
                sv.sv_apply_circuit(s, c)
            sv.sv_sync(s)
            times.append(time.perf_counter() - t)
        best.append(min(times))
    s.free()
    assert best[0] < 1.5 * best[1], best
