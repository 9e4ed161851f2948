"""Schedules on states of up to 12 qubits, which run many gates per launch (one cluster holds
the state): every width, gate kind and target position against the oracle and against the
pass-per-gate kernels, and the schedules captured in a CUDA graph."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
TOL = {0: 1e-5, 1: 1e-12}     # the library's stated max-abs amplitude errors


def _mixed(n, count, rng):
    """(targets, U): dense, diagonal, permutation and controlled gates on unsorted targets."""
    gates = []
    for i in range(count):
        k = int(rng.integers(1, min(5, n) + 1))
        tg = tuple(int(t) for t in rng.choice(n, size=k, replace=False))
        d = 1 << k
        kind = i % 4
        if kind == 0:
            u = np.array(W.haar_unitary(d, rng)).reshape(d, d)
        elif kind == 1:
            u = np.diag(np.where(rng.random(d) < 0.4, 1.0, np.exp(1j * rng.uniform(0, 6, d))))
        elif kind == 2:
            u = np.zeros((d, d), dtype=np.complex128)
            u[np.arange(d), rng.permutation(d)] = np.where(rng.random(d) < 0.5, 1.0, np.exp(1j * rng.uniform(0, 6, d)))
        else:                                     # controlled on its highest local bit
            u = np.eye(d, dtype=np.complex128)
            h = d // 2
            u[h:, h:] = np.array(W.haar_unitary(h, rng)).reshape(h, h) if h > 1 else np.exp(0.7j)
        gates.append((tg, u))
    return gates


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 4, 5, 6, 8, 9, 11, 12, 13])
def test_small_states_match_the_oracle_and_the_passes(gpu, dtype, n):
    """13 qubits: the first width that runs pass by pass."""
    sv = gpu
    import torch
    rng = np.random.default_rng(700 + n)
    gates = _mixed(n, 40, rng)                    # more than one launch's parameters at k = 5
    psi0 = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi0 = (psi0 / np.linalg.norm(psi0)).astype(np.complex64 if dtype == 0 else np.complex128)
    ref = oracle.run(psi0.astype(np.complex128), gates)
    for max_k in (0, 3):
        got = []
        for policy in (0, sv.SV_POLICY_NO_TENSOR_CORES):
            s = sv.sv_alloc(n, dtype, stream=torch.cuda.current_stream())
            sv.sv_set_policy(s, policy)
            sv.sv_set_state(s, psi0)
            c = sv.sv_fuse(gates, n, max_k)
            rep = sv.sv_apply_circuit(s, c)
            got.append((sv.sv_get_state(s), rep))
            s.free()
            assert np.max(np.abs(got[-1][0] - ref)) < TOL[dtype], (n, max_k, policy)
        a, b = got[0][1], got[1][1]
        if n <= 12 and not (dtype == 1 and n >= 11):   # there the flag changes the schedule
            assert (a["passes"], a["bytes"], a["max_k_used"]) == (b["passes"], b["bytes"], b["max_k_used"])


def test_untouched_amplitudes_come_back_bit_for_bit(gpu):
    sv = gpu
    rng = np.random.default_rng(5)
    n = 12
    u = np.eye(8, dtype=np.complex128)
    u[6:, 6:] = np.array(W.haar_unitary(2, rng)).reshape(2, 2)       # controls: local bits 1, 2
    psi0 = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)).astype(np.complex64)
    for tg in ((0, 3, 11), (11, 10, 2), (4, 0, 1)):
        s = sv.sv_alloc(n, 0)
        sv.sv_set_state(s, psi0)
        sv.sv_apply_circuit(s, sv.sv_fuse([(tg, u)], n, 0))
        got = sv.sv_get_state(s)
        s.free()
        i = np.arange(1 << n)
        out = ((i >> tg[1]) & (i >> tg[2]) & 1) == 0
        assert np.array_equal(got[out].view(np.uint32), psi0[out].view(np.uint32))


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n", [10, 14])
def test_a_captured_schedule_replays(gpu, dtype, n):
    sv = gpu
    import torch
    gl = sv.gates_from_specs(W.brickwork(n, 6))
    ref = oracle.simulate(n, W.brickwork(n, 6), x=3)
    c = sv.sv_fuse(gl, n, 2)
    buf = torch.empty(1 << n, device="cuda", dtype=torch.complex64 if dtype == 0 else torch.complex128)
    st = torch.cuda.Stream()
    s = sv.sv_alloc(n, dtype, dev_buf=buf, stream=st)
    sv.sv_set_basis(s, 3)
    sv.sv_apply_circuit(s, c)                     # one-time setup outside the capture
    sv.sv_sync(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        sv.sv_set_basis(s, 3)
        sv.sv_apply_circuit(s, c)
    for _ in range(2):
        buf.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert np.max(np.abs(buf.cpu().numpy() - ref)) < TOL[dtype]
    s.free()
